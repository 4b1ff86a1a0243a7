"""The U-Net convolution's routes on the GPU against FP64, as in
test_gpu_unet.py (inputs on BF16 values, so only FP32 sums differ; bound
4 sqrt(K) 2^-24 of the largest output, K the contraction length): halo
blocks (32 and 64 input channels, rows of 128, 64 and 32 cells, strips and
plane groups that end past the grid, channel tiles of 32 to 96) and sums split
over slices of the taps (few cell tiles, one sample to several)."""
import numpy as np
import pytest

import oracle.unet as U
from test_gpu_unet import _conv_case, _dev, _first, _need_gpu, _sum_tol, _w5

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [
    (3, 4, 8, 128, 32, 32),      # halo, one row per tile
    (5, 4, 8, 64, 64, 64),       # halo, tiles across rows
    (3, 8, 16, 32, 32, 96),
    (5, 4, 16, 32, 64, 32),
    (1, 8, 16, 128, 64, 32),
    (2, 4, 4, 8, 256, 512),      # split, two cell tiles
    (1, 2, 2, 2, 64, 32),        # split, a part of one tile
    (7, 1, 1, 4, 96, 160),
]


@pytest.mark.parametrize("case", CASES)
def test_conv_routes_match_fp64(case):
    _need_gpu()
    from paper_2606_16765_gb300 import unet as N
    B, nz, ny, nx, cin, cout = case
    x, w, g = _conv_case(sum(case), B, nz, ny, nx, cin, cout)
    y = torch.full((B, nz, ny, nx, cout), float("nan"), device="cuda")
    gx = torch.full((B, nz, ny, nx, cin), float("nan"), device="cuda")
    N.conv3_forward(_dev(x), _dev(w), y)
    N.conv3_backward_data(_dev(g), _dev(w), gx)
    ref = np.moveaxis(U.conv3(_first(x), _w5(w)), 1, -1)
    rgx = np.moveaxis(U.conv3_backward(_first(x), _w5(w), _first(g))[0], 1, -1)
    ey = np.abs(y.cpu().numpy() - ref).max() / np.abs(ref).max()
    ex = np.abs(gx.cpu().numpy() - rgx).max() / np.abs(rgx).max()
    print(f"conv {case}: forward {ey:.2e}, input gradient {ex:.2e}")
    assert ey < _sum_tol(27 * cin) and ex < _sum_tol(27 * cout)


@pytest.mark.parametrize("case", [(2, 4, 8, 16, 64, 64), (1, 2, 2, 4, 128, 192), (3, 4, 4, 8, 64, 320), (2, 4, 4, 8, 192, 64)])
def test_weight_gradient_with_64_channel_rows(case):
    """Weight gradients whose operands are copied 64 channels at a time (both
    counts multiples of 64), tiles past the batch and channel tiles included."""
    _need_gpu()
    from paper_2606_16765_gb300 import unet as N
    B, nz, ny, nx, cin, cout = case
    x, w, g = _conv_case(sum(case), B, nz, ny, nx, cin, cout)
    gw = torch.full((cout, cin, 27), float("nan"), device="cuda")
    N.conv3_backward_weights(_dev(x), _dev(g), gw)
    ref = U.conv3_backward(_first(x), _w5(w), _first(g))[1].reshape(cout, cin, 27)
    err = np.abs(gw.cpu().numpy() - ref).max() / np.abs(ref).max()
    print(f"weight gradient {case}: {err:.2e}")
    assert err < _sum_tol(B * nz * ny * nx)
