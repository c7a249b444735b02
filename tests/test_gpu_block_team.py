"""Block teams (1, 2 and 4 lanes per block, and the idle lanes beyond) on
blocks that touch each other, against the FP64 oracle.

Blocks packed side by side, so that every kind of pair is in force: a pusher on
its own block, a pusher on another block, a corner in another block.  The bars
and the conditioning of tests/_common.py apply (softer contact); the widths
differ only in the order in which forces between blocks are summed."""
import numpy as np
import pytest
import torch

from oracle import stamp_oracle as O
from paper_2310_01775_gb300 import workloads as W

from _common import Reference

pytestmark = pytest.mark.gpu

WIDTHS = {1: (1, 2, 4), 2: (2, 4, 8, 16), 3: (8, 16, 32), 4: (8, 16, 32)}


def packed_scene(nb):
    base = np.array([[-0.5, -0.5], [0.5, -0.5], [-0.5, 0.5], [0.5, 0.5]])[:nb] * 0.104
    init = np.concatenate([base, np.array([[0.02], [-0.03], [0.01], [0.04]])[:nb]], 1)
    goal = init + np.array([0.05, -0.03, 0.1])
    f = lambda x: x.astype(np.float32).astype(np.float64)  # noqa: E731
    return f(init), f(goal)


@pytest.mark.parametrize("C", [1, 25])
@pytest.mark.parametrize("nb,lanes", [(nb, 0) for nb in WIDTHS] +
                         [(nb, w) for nb, ws in WIDTHS.items() for w in ws])
def test_every_team_width_on_touching_blocks(nb, lanes, C):
    from paper_2310_01775_gb300 import stamp as S
    N, H, T, seed, it = 37, 1, 50, 3, 2       # ragged at every width
    P = W.params("pusher3_h6", n_blocks=nb, H=H, T=T, ckpt_every=C, k_contact=1e3, c_contact=10.0)
    P = {k: (float(np.float32(v)) if isinstance(v, float) else v) for k, v in P.items()}
    init, goal = packed_scene(nb)
    M, _, D = O.dims(P)
    theta = O.init_theta(seed, N, D).astype(np.float32)
    prob = S.Problem(P, init, goal, N, torch.cuda.current_stream().cuda_stream)
    prob.set_lanes(lanes, lanes)
    th = torch.tensor(theta, device="cuda")
    cost, fin = torch.empty(N, device="cuda"), torch.empty(N, prob.S, device="cuda")
    tape = torch.empty(prob.n_ckpt + 1, N, prob.S, device="cuda")
    grads = []
    prob.rollout_fwd(th, N, seed, it, 0, cost, fin)
    prob.read_tape(N, tape)
    for mode in (S.STAMP_ADJ_AUTO, S.STAMP_ADJ_SEQUENTIAL):   # stored rows, segment recompute
        prob.set_adjoint_mode(mode)
        grads.append(torch.empty(N, D, device="cuda"))
        prob.rollout_adjoint(th, N, seed, it, grads[-1])
    prob.sync()
    prob.close()
    ref = Reference(theta, P, init, goal, O.gumbel_noise(seed, it, N, H, M), C=C)
    if nb > 1:   # the blocks do meet
        xy = O.rollout(theta.astype(np.float64), P, init, goal, O.gumbel_noise(seed, it, N, H, M),
                       record=True)[2][..., :2]
        gap = min(np.linalg.norm(xy[:, :, a] - xy[:, :, b], axis=-1).min()
                  for a in range(nb) for b in range(a))
        assert gap < 0.1
    t = tape.cpu().numpy().transpose(1, 0, 2).reshape(N, -1, nb, 6)
    for g in grads:
        ref.check(t, fin.cpu().numpy(), cost.cpu().numpy(), g.cpu().numpy(), min_frac=0.3)
