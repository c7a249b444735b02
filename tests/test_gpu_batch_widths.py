"""Batched solves at every team width the batch accepts, and at the widths its
autotuner picks, against the same instances solved alone.

A class whose launch leaves particles out keeps their old costs and gradients
(zero at first), so every particle is compared, and the last iteration's
gradients too.  Bars as in tests/test_gpu_batch.py: 1e-5 after three
iterations (the same kernel bodies, rounding differently where the compiler
fuses differently); the gradients, which the contact dynamics amplify, to 1e-3
of the largest."""
import numpy as np
import pytest
import torch

from paper_2310_01775_gb300 import workloads as W

pytestmark = pytest.mark.gpu

T, ITERS, LR = 50, 3, 1e-2
PHYSICS = dict(W.PHYSICS, T=T, k_contact=1e3, c_contact=10.0)   # reproducible over whole plans
SHAPES = [(1, 2, 37), (2, 3, 64), (3, 2, 100), (4, 2, 45), (1, 4, 200), (3, 3, 33), (2, 1, 150), (4, 1, 70)]
WIDTHS = {1: (1, 2, 4), 2: (2, 4, 8, 16), 3: (8, 16, 32), 4: (8, 16, 32)}


def _batch():
    from paper_2310_01775_gb300 import stamp as S
    insts = []
    for g, (nb, H, N) in enumerate(SHAPES):
        init, goal = W.scene({"n_blocks": nb}, 40 + g)
        insts.append({"n_blocks": nb, "H": H, "N": N, "seed": 1000 + g, "init": init, "goal": goal})
    return S.Batch(PHYSICS, insts, torch.cuda.current_stream().cuda_stream), insts


def _alone(d, lanes, C):
    """theta, lowest hard cost and the last iteration's gradient of one instance."""
    from paper_2310_01775_gb300 import stamp as S
    P = dict(PHYSICS, n_blocks=d["n_blocks"], H=d["H"], ckpt_every=C)
    prob = S.Problem(P, d["init"], d["goal"], d["N"], torch.cuda.current_stream().cuda_stream)
    prob.set_lanes(lanes, lanes)
    prob.set_adjoint_mode(S.STAMP_ADJ_SEQUENTIAL)
    th, before = torch.empty(d["N"], prob.D, device="cuda"), torch.empty(d["N"], prob.D, device="cuda")
    cost, grad = torch.empty(d["N"], device="cuda"), torch.empty(d["N"], prob.D, device="cuda")
    prob.solve(d["N"], ITERS - 1, 0, d["seed"], LR, None, before)
    prob.rollout_fwd(before, d["N"], d["seed"], ITERS - 1, 0, cost)
    prob.rollout_adjoint(before, d["N"], d["seed"], ITERS - 1, grad)
    prob.solve(d["N"], ITERS, 0, d["seed"], LR, None, th, cost)
    prob.sync()
    prob.close()
    return th, float(cost.min()), grad


def _compare(b, insts):
    res = b.results()
    for g, d in enumerate(insts):
        lanes, _, C = b.get_config(d["n_blocks"])
        want, best, grad = _alone(d, lanes, C)
        theta, got = torch.empty_like(want), torch.empty_like(want)
        b.read_theta(g, theta)
        b.read_grad(g, got)
        assert float((theta - want).abs().max()) <= 1e-5, (g, lanes)
        assert float((got - grad).abs().max()) <= 1e-3 * float(grad.abs().max()), (g, lanes)
        assert abs(res["best_cost"][g] - best) <= 1e-5 * max(best, 1e-6), (g, lanes)


@pytest.mark.parametrize("cta,C", [(32, 25), (64, 1), (128, 5)])
@pytest.mark.parametrize("nb,lanes", [(nb, w) for nb, ws in WIDTHS.items() for w in ws])
def test_every_accepted_width(nb, lanes, cta, C):
    b, insts = _batch()
    b.set_config(nb, lanes, cta, C)
    b.solve(ITERS, LR)
    _compare(b, insts)
    b.close()


def test_autotuned_widths():
    b, insts = _batch()
    b.autotune(1)
    b.solve(ITERS, LR)
    _compare(b, insts)
    b.close()
