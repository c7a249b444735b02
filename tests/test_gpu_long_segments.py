"""The sequential reverse sweep of checkpoint segments that are long for the shared
memory of many narrow teams: the automatic width takes two lanes or one per block
from some particle count on, and a CTA then holds more teams' segments than at
the width it takes for a few particles.  Every row is the few particles' row."""
import pytest
import torch

from oracle import stamp_oracle as O
from paper_2310_01775_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,N,T", [(1, 9800, 200), (2, 5000, 200), (2, 9800, 100), (3, 4900, 150), (4, 2600, 200)])
def test_sequential_sweep_of_one_segment_per_push(nb, N, T):
    from paper_2310_01775_gb300 import stamp as S
    P = W.params("pusher3_h6", n_blocks=nb, H=1, T=T, ckpt_every=T)
    init, goal = W.scene(P, 0)
    few, seed, it = 40, 5, 1
    D = O.dims(P)[2]
    theta = torch.tensor(O.init_theta(seed, N, D), dtype=torch.float32, device="cuda")
    prob = S.Problem(P, init, goal, N, torch.cuda.current_stream().cuda_stream)
    prob.set_adjoint_mode(S.STAMP_ADJ_SEQUENTIAL)

    def gradient(n):
        th = theta[:n].contiguous()
        cost, g = torch.empty(n, device="cuda"), torch.empty(n, D, device="cuda")
        prob.rollout_fwd(th, n, seed, it, 0, cost)
        prob.rollout_adjoint(th, n, seed, it, g)
        prob.sync()
        return g

    g = gradient(N)
    assert torch.isfinite(g).all()
    assert torch.equal(g[:few], gradient(few))
    prob.close()
