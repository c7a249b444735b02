"""The surrogate's rollout on every tile shape and its selection at its edges."""
import numpy as np
import pytest
import torch

from paper_2310_01775_gb300 import workloads as W
from test_gpu_surrogate import _packed, _random_net, _S, _stream

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,H", [(1, 1), (2, 3), (3, 6)])
def test_plans_do_not_depend_on_how_many_there_are(nb, H):
    """Tiles of 32 and 64 plans (two CTAs each) and of 128: costs and gradients of
    the first plans have the same bits, with and without the gradient."""
    S = _S()
    P = dict(W.params("pusher3_h6"), n_blocks=nb, H=H)
    init, goal = W.scene(P, 2)
    n_max = 128 * 40
    prob = S.Problem(P, init, goal, n_max, _stream())
    sur = S.Surrogate(P, n_max, n_max, _stream())
    sur.set_params(_packed(_random_net(nb, 5)))
    theta = torch.tensor(W.random_theta(n_max, prob.D, 4), device="cuda")
    pair = torch.cuda.get_device_properties(0).multi_processor_count // 2
    ref = None
    for N in (n_max, pair * 64, pair * 32 + 1, pair * 32, 33, 1):
        cost = torch.full((N,), float("nan"), device="cuda")
        only = torch.full((N,), float("nan"), device="cuda")
        grad = torch.full((N, prob.D), float("nan"), device="cuda")
        sur.rollout(prob, theta, N, 3, 9, cost, grad)
        sur.rollout(prob, theta, N, 3, 9, only)
        sur.sync()
        if ref is None:
            ref = cost, grad
            assert torch.isfinite(cost).all() and torch.isfinite(grad).all()
        assert torch.equal(cost, ref[0][:N]) and torch.equal(only, cost), N
        assert torch.equal(grad, ref[1][:N]), N
    sur.close()
    prob.close()


@pytest.mark.parametrize("n_cand,N,copies", [(1, 1, 1), (4096, 4096, 1), (20001, 777, 1), (6000, 4096, 500),
                                             (6000, 1, 6000)])
def test_selection_orders_ties_by_index(n_cand, N, copies):
    """The N lowest costs in order, equal ones (copies of a plan) by index."""
    S = _S()
    P = W.params("pusher1_h4")
    init, goal = W.scene(P, 2)
    prob = S.Problem(P, init, goal, N, _stream())
    sur = S.Surrogate(P, n_cand, N, _stream())
    sur.set_params(_packed(_random_net(1, 5)))
    plans = torch.tensor(W.random_theta((n_cand + copies - 1) // copies, prob.D, 4), device="cuda")
    cand = plans.repeat(copies, 1)[:n_cand].contiguous()
    cost = torch.empty(n_cand, device="cuda")
    sur.rollout(prob, cand, n_cand, 0, -1, cost)
    theta = torch.empty(N, prob.D, device="cuda")
    index = torch.empty(N, dtype=torch.int32, device="cuda")
    sur.screen(prob, cand, n_cand, N, theta, index)
    sur.sync()
    want = np.lexsort((np.arange(n_cand), cost.cpu().numpy()))[:N]
    assert np.array_equal(index.cpu().numpy(), want)
    assert torch.equal(theta, cand[torch.tensor(want, device="cuda")])
    sur.close()
    prob.close()
