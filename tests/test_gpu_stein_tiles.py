"""Stein steps at the edges of their tiles and of the rules that pick a kernel,
against the FP64 oracle: 64-particle distance tiles, 32-row tiles of the sum,
32-column slots, the one-CTA step (N <= 64), eight rows per warp (N >= 1921 on
152 SMs), the structured kernel's 16-row tiles.  Bounds as in
tests/test_gpu_svgd.py: 1e-5 of the summed terms' magnitude."""
import numpy as np
import pytest
import torch

from oracle import stamp_oracle as O
from paper_2310_01775_gb300 import workloads as W

from test_gpu_svgd import make_problem, term_scale

pytestmark = pytest.mark.gpu


def check(theta, g, h, phi):
    h_ref = O.median_bandwidth(theta) if len(theta) > 1 else 1.0
    assert abs(h - h_ref) <= 1e-5 * h_ref
    err = np.abs(phi - O.stein_direction(theta, g, h_ref))
    assert (err <= 1e-5 * term_scale(theta, g, h_ref) + 1e-9).all()


@pytest.mark.parametrize("N", [1, 2, 63, 64, 65, 127, 129, 2000])
@pytest.mark.parametrize("nb,H", [(1, 1), (1, 16)])   # D = 6 and 96
def test_rbf_step(N, nb, H):
    prob, _ = make_problem(N, n_blocks=nb, H=H)
    theta, g = W.random_theta(N, prob.D, N + H), W.random_normal((N, prob.D), N + H + 1)
    th, gr = torch.tensor(theta, device="cuda"), torch.tensor(g, device="cuda")
    m, v = torch.zeros_like(th), torch.zeros_like(th)
    h, phi = torch.zeros(1, device="cuda"), torch.zeros_like(th)
    prob.svgd_step(th, gr, N, m, v, 1, 1e-2, 0, h, phi)
    prob.sync()
    prob.close()
    check(theta, g, float(h), phi.cpu().numpy())


@pytest.mark.parametrize("N,D", [(65, 1), (33, 31), (65, 32), (64, 33), (130, 65), (96, 97), (70, 288)])
def test_column_slots(N, D):
    """Any D, through the allocation-free step (the same kernels, one share)."""
    from paper_2310_01775_gb300 import stamp as S
    theta, g = W.random_theta(N, D, D), W.random_normal((N, D), D + 1)
    th, gr = torch.tensor(theta, device="cuda"), torch.tensor(g, device="cuda")
    m, v = torch.zeros_like(th), torch.zeros_like(th)
    h, phi = torch.zeros(1, device="cuda"), torch.zeros_like(th)
    S.stamp_svgd_step_noalloc(th, gr, N, D, m, v, 1, 1e-2, 0, h, phi,
                              torch.cuda.current_stream().cuda_stream)
    check(theta, g, float(h), phi.cpu().numpy())


@pytest.mark.parametrize("N,nb,H", [(2, 1, 1), (15, 1, 2), (17, 2, 3), (33, 4, 16)])
def test_structured_step(N, nb, H):
    prob, P = make_problem(N, n_blocks=nb, H=H)
    prob.set_svgd_kernel(1)
    theta, g = W.random_theta(N, prob.D, N), W.random_normal((N, prob.D), N + 1)
    th, gr = torch.tensor(theta, device="cuda"), torch.tensor(g, device="cuda")
    m, v = torch.zeros_like(th), torch.zeros_like(th)
    h, phi = torch.zeros(1, device="cuda"), torch.zeros_like(th)
    prob.svgd_step(th, gr, N, m, v, 1, 1e-2, 0, h, phi)
    prob.sync()
    prob.close()
    ref = O.stein_direction_structured(theta.astype(np.float64), g.astype(np.float64), P)
    ref = ref[0] if isinstance(ref, tuple) else ref
    assert np.abs(phi.cpu().numpy() - ref).max() <= 1e-4 * np.abs(ref).max()


@pytest.mark.parametrize("N,nb,H", [(1921, 1, 6), (2113, 4, 7), (1921, 4, 16)])   # D = 36, 126, 288
def test_many_particles(N, nb, H):
    """Eight rows per warp; a shard of the rows (ragged, not at a tile's edge) sums
    as all rows do."""
    prob, _ = make_problem(N, n_blocks=nb, H=H)
    theta, g = W.random_theta(N, prob.D, N + H), W.random_normal((N, prob.D), N + H + 1)
    th, gr = torch.tensor(theta, device="cuda"), torch.tensor(g, device="cuda")
    h, phi = torch.zeros(1, device="cuda"), torch.zeros_like(th)
    m, v = torch.zeros_like(th), torch.zeros_like(th)
    a = th.clone()
    prob.svgd_step(a, gr, N, m, v, 1, 1e-2, 0, h, phi)
    prob.sync()
    check(theta, g, float(h), phi.cpu().numpy())
    row0, rows = 130, N - 161
    part = th[row0:row0 + rows].clone()
    m, v = torch.zeros_like(part), torch.zeros_like(part)
    prob.svgd_step_rows(th, gr, N, row0, rows, part, m, v, 1, 1e-2, 0)
    prob.sync()
    prob.close()
    assert torch.equal(part, a[row0:row0 + rows])
