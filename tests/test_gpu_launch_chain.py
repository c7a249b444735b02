"""The launch chains captured into a CUDA graph: a replay on new inputs gives the
bits of direct calls (every kernel waits for the one before it)."""
import pytest
import torch

from paper_2310_01775_gb300 import workloads as W
from test_gpu_surrogate import _packed, _random_net

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,H,C,N,kind", [(1, 2, 1, 200, 0), (3, 2, 25, 300, 0), (2, 3, 25, 2000, 0), (1, 2, 1, 150, 1)])
def test_replay_equals_direct_calls(nb, H, C, N, kind):
    from paper_2310_01775_gb300 import stamp as S
    P = dict(W.params("pusher3_h6"), n_blocks=nb, H=H, T=50, ckpt_every=C)
    init, goal = W.scene(P, 2)
    st = torch.cuda.Stream()
    prob = S.Problem(P, init, goal, N, st.cuda_stream)
    prob.set_svgd_kernel(kind)
    sur = S.Surrogate(P, max(N, 256), N, st.cuda_stream)
    sur.set_params(_packed(_random_net(nb, 3)))
    sets = [torch.tensor(W.random_theta(N, prob.D, s), device="cuda") for s in (1, 2, 3)]
    theta, m, v = (torch.zeros(N, prob.D, device="cuda") for _ in range(3))
    cost, scost, h = torch.zeros(N, device="cuda"), torch.zeros(N, device="cuda"), torch.zeros(1, device="cuda")
    final = torch.zeros(N, prob.S, device="cuda")
    grad, sgrad, phi = (torch.zeros(N, prob.D, device="cuda") for _ in range(3))

    def chain():
        prob.rollout_fwd(theta, N, 5, 3, 0, cost, final)
        prob.rollout_adjoint(theta, N, 5, 3, grad)
        sur.rollout(prob, theta, N, 5, 3, scost, sgrad)
        prob.svgd_step(theta, sgrad, N, m, v, 1, 1e-2, 0, h, phi)

    def outputs(x, call):
        with torch.cuda.stream(st):
            theta.copy_(x), m.zero_(), v.zero_()
            call()
            st.synchronize()
            return [t.clone() for t in (cost, final, grad, scost, sgrad, h, phi, theta)]

    torch.cuda.synchronize()
    direct = [outputs(x, chain) for x in sets]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        chain()
    for x, want in zip(sets, direct):
        for a, b in zip(outputs(x, graph.replay), want):
            assert torch.equal(a, b)
    prob.sync()
    sur.close()
    prob.close()
