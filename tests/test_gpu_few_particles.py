"""Which kernels a Stein step of few particles runs, by its particles and columns:
one CTA where that is the shorter, the general kernels elsewhere, with the same
bits.  Where a solve can run the bandwidth beside its rollouts the line is lower."""
import pytest
import torch

from oracle import stamp_oracle as O
from paper_2310_01775_gb300 import workloads as W

from test_gpu_svgd import make_problem

pytestmark = pytest.mark.gpu


def pairwise_launches(prob, call):
    prob.set_profiling(True)
    call()
    prob.sync()
    n = prob.kernel_times()["pairwise"][1]
    prob.set_profiling(False)
    return n


# (blocks, H, N): the columns are H (4 blocks + 2)
@pytest.mark.parametrize("nb,H,N,one_cta", [(1, 2, 2, True), (4, 16, 32, True), (4, 16, 33, False),
                                            (3, 6, 41, True), (3, 6, 42, False), (1, 4, 64, True),
                                            (1, 5, 58, True), (1, 5, 59, False), (4, 16, 64, False),
                                            (1, 2, 65, False)])
def test_step(nb, H, N, one_cta):
    prob, P = make_problem(N, n_blocks=nb, H=H)
    D = prob.D
    th0 = torch.tensor(W.random_theta(N, D, 3 + N), device="cuda")
    g = torch.tensor(W.random_normal((N, D), 4 + N), device="cuda")

    def state():
        return [th0.clone(), torch.zeros_like(th0), torch.zeros_like(th0), torch.zeros_like(th0)]

    (th, m, v, phi), (th2, m2, v2, phi2) = state(), state()
    h, h2 = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
    launches = pairwise_launches(prob, lambda: prob.svgd_step(th, g, N, m, v, 3, 1e-2, 0, h, phi))
    assert launches == (0 if one_cta else 1)
    prob.svgd_step_rows(th0, g, N, 0, N, th2, m2, v2, 3, 1e-2, 0, h2, phi2)   # the general kernels
    prob.sync()
    prob.close()
    for a, b in ((th, th2), (m, m2), (v, v2), (phi, phi2), (h, h2)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("nb,H,N,one_cta", [(1, 2, 32, True), (1, 2, 33, False), (3, 6, 24, True), (3, 6, 25, False)])
def test_solve(nb, H, N, one_cta):
    prob, P = make_problem(N, n_blocks=nb, H=H, T=25)
    th0 = torch.tensor(O.init_theta(7, N, prob.D), dtype=torch.float32, device="cuda")
    out, alone = torch.empty_like(th0), torch.empty_like(th0)
    launches = pairwise_launches(prob, lambda: prob.solve(N, 3, 1, 7, 1e-2, th0, out))
    assert launches == (0 if one_cta else 3)
    prob.set_overlap(False)
    prob.solve(N, 3, 1, 7, 1e-2, th0, alone)
    prob.close()
    assert torch.equal(out, alone)
