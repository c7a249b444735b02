"""The sweep of a solve's last hard rollout, which left no per-substep rows beside
its checkpoints: the sweep that reads rows gives what it gives after the same
rollout made by itself, not what an iteration's rows would."""
import pytest
import torch

from oracle import stamp_oracle as O
from paper_2310_01775_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("nb", [1, 3])
def test_sweep_after_a_solve(nb, weighted):
    from paper_2310_01775_gb300 import stamp as S
    P = W.params("pusher3_h6", n_blocks=nb, H=2, T=50, ckpt_every=25)
    init, goal = W.scene(P, 0)
    N, seed = 70, 4
    D = O.dims(P)[2]
    theta = torch.tensor(O.init_theta(1, N, D), dtype=torch.float32, device="cuda")
    out, cost = torch.empty_like(theta), torch.empty(N, device="cuda")
    got, want = torch.empty_like(theta), torch.empty_like(theta)
    prob = S.Problem(P, init, goal, N, torch.cuda.current_stream().cuda_stream)
    prob.set_adjoint_mode(S.STAMP_ADJ_REPLAY)
    prob.set_dsvgd(weighted)
    prob.solve(N, 2, 1, seed, 1e-2, theta, out)
    for _ in range(2):
        prob.rollout_adjoint(out, N, seed, -1, got)
    prob.rollout_fwd(out, N, seed, -1, 1, cost)
    prob.rollout_adjoint(out, N, seed, -1, want)
    prob.sync()
    prob.close()
    assert bool((want != 0).any())
    assert torch.equal(got, want)
