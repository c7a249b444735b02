"""The MLP at the edges of its tiles and widths: the forward that packs its
input and writes its output itself, the weight gradients on the saved tiles."""
import numpy as np
import pytest
import torch

from paper_2310_01775_gb300 import workloads as W
from test_gpu_mlp import packed, rounded_backward

pytestmark = pytest.mark.gpu
WIDTHS = [(26, 9), (32, 16), (1, 1)]


def _net(n_in, n_out, rows, train_rows=0):
    from paper_2310_01775_gb300 import stamp as S
    params = W.mlp_init([n_in, 256, 256, 256, n_out], 31)
    net = S.MLP(n_in, n_out, rows, train_rows, torch.cuda.current_stream().cuda_stream)
    net.set_params(torch.tensor(packed(params), device="cuda"))
    return net, params


@pytest.mark.parametrize("n_in,n_out", WIDTHS)
@pytest.mark.parametrize("rows", [1, 129, 20011])
def test_rows_do_not_depend_on_their_tile(n_in, n_out, rows):
    """More tiles than SMs (a CTA takes several), a last tile of few rows, and a
    y inside x's storage give each row the bits it has in a call of its own."""
    net, _ = _net(n_in, n_out, rows)
    x = torch.rand(rows, n_in, device="cuda") * 2 - 1
    y = torch.full((rows, n_out), float("nan"), device="cuda")
    net.forward(x, rows, y)
    part = torch.empty_like(y)
    for r0 in range(0, rows, 7001):
        n = min(7001, rows - r0)
        net.forward(x[r0:r0 + n].contiguous(), n, part[r0:r0 + n])
    net.sync()
    assert torch.equal(y, part)
    if n_out <= n_in:
        flat = x.clone().flatten()
        inside = flat[:rows * n_out].view(rows, n_out)
        net.forward(flat.view(rows, n_in), rows, inside)
        net.sync()
        assert torch.equal(inside, y)
    net.close()


@pytest.mark.parametrize("n_in,n_out", WIDTHS[1:])
@pytest.mark.parametrize("rows", [129, 3600])
def test_weight_gradients_at_the_widths_of_the_operands(n_in, n_out, rows):
    """Against float64 with the kernel's bfloat16 storage points; the bar is the
    one of the backward test (a rounding of the stored dz moves it by 2^-9)."""
    net, params = _net(n_in, n_out, rows, rows)
    rng = np.random.default_rng(rows)
    x, dy = rng.uniform(-1, 1, size=(rows, n_in)), rng.standard_normal((rows, n_out))
    y = torch.empty(rows, n_out, device="cuda")
    dp = torch.full((net.n_params,), float("nan"), device="cuda")
    net.forward_saved(torch.tensor(x, dtype=torch.float32, device="cuda"), rows, y, 0)
    net.backward(torch.tensor(dy, dtype=torch.float32, device="cuda"), rows, 0, None, dp)
    net.sync()
    net.close()
    dp, off = dp.cpu().numpy(), 0
    for gW, gb in rounded_backward(params, x, dy)[0]:
        ref = np.concatenate([gW.ravel(), gb])
        assert np.abs(dp[off:off + ref.size] - ref).max() <= 2e-2 * np.abs(ref).max(), off
        off += ref.size
