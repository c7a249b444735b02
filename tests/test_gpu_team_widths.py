"""A rollout's results do not depend on how many particles are rolled out with it:
the lanes of a team are picked by that count, and every width gives the same
bits, on blocks that touch each other too (so a set's shards are the set)."""
import pytest
import torch

from oracle import stamp_oracle as O
from paper_2310_01775_gb300 import workloads as W

from test_gpu_block_team import packed_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [1, 25])
@pytest.mark.parametrize("nb,widths", [(1, (1, 2, 4)), (2, (2, 4, 8, 16)), (3, (8, 16, 32)), (4, (8, 16, 32))])
def test_the_width_does_not_change_the_bits(nb, widths, C):
    """Costs, states and gradients of touching blocks at every width; automatic
    widths too, at a count that takes one lane per block for up to three blocks."""
    from paper_2310_01775_gb300 import stamp as S
    P = W.params("pusher3_h6", n_blocks=nb, H=1, T=50, ckpt_every=C)
    init, goal = packed_scene(nb)
    N, big, seed, it = 149, {1: 9800, 2: 9800, 3: 4900, 4: 2600}[nb], 3, 2
    D = O.dims(P)[2]
    theta = torch.tensor(O.init_theta(seed, big, D), dtype=torch.float32, device="cuda")
    prob = S.Problem(P, init, goal, big, torch.cuda.current_stream().cuda_stream)
    prob.set_adjoint_mode(S.STAMP_ADJ_REPLAY)

    def outputs(n, lanes):
        prob.set_lanes(lanes, lanes)
        th = theta[:n].contiguous()
        cost, fin, g = torch.empty(n, device="cuda"), torch.empty(n, prob.S, device="cuda"), torch.empty(n, D, device="cuda")
        prob.rollout_fwd(th, n, seed, it, 0, cost, fin)
        prob.rollout_adjoint(th, n, seed, it, g)
        prob.sync()
        return [t[:N].clone() for t in (cost, fin, g)]

    want = outputs(N, widths[-1])
    for got in [outputs(N, w) for w in (0, *widths)] + [outputs(big, 0)]:
        for a, b in zip(got, want):
            assert torch.equal(a, b)
    prob.close()
