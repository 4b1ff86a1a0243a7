"""Which kernel takes a convolution call, and that it is right there: halo blocks
over rows of 128, 64, 32 and 16 cells, weights in stages of three taps and of one,
one and two accumulator sets, shifted copies, and split sums.  Sizes lie well
inside their route's range (it depends on the number of SMs).  Against FP64 with
the bound of test_gpu_conv_routes.py (4 sqrt(K) 2^-24 of the largest output)."""
import ctypes as C

import numpy as np
import pytest

import oracle.unet as U
from test_gpu_unet import _conv_case, _dev, _first, _need_gpu, _sum_tol, _w5

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

COPIES, HALO, SPLIT = 0, 1, 2
# B, nz, ny, nx, cin, cout: route and, for halo blocks, taps per stage and accumulator sets
CASES = [
    ((2, 8, 16, 128, 32, 32), HALO, 3, 2),
    ((4, 16, 16, 64, 64, 64), HALO, None, 2),
    ((8, 8, 16, 32, 32, 64), HALO, 3, 2),
    ((16, 8, 16, 16, 64, 64), HALO, 3, 2),
    ((16, 16, 8, 16, 32, 32), HALO, 3, 2),
    ((2, 8, 32, 64, 64, 256), HALO, 1, 1),
    ((2, 16, 16, 64, 32, 256), HALO, 3, 1),
    ((4, 8, 16, 32, 96, 64), COPIES, None, None),
    ((2, 4, 4, 8, 256, 128), SPLIT, None, None),
    ((3, 2, 2, 2, 64, 32), SPLIT, None, None),
]


@pytest.mark.parametrize("case,route,taps,sets", CASES)
def test_plan_and_result(case, route, taps, sets):
    _need_gpu()
    from paper_2606_16765_gb300 import unet as N
    B, nz, ny, nx, cin, cout = case
    x, w, g = _conv_case(sum(case), B, nz, ny, nx, cin, cout)
    xd = _dev(x)
    got = (C.c_int32 * 5)()
    assert N.lib().unet_conv3_route(C.c_void_p(xd.data_ptr()), B, nx, ny, nz, cin, cout, got) == 0
    print(f"conv {case}: route {got[0]}, {got[1]} parts, channel tile {got[2]}, {got[3]} taps a stage, {got[4]} sets")
    assert got[0] == route and (taps is None or got[3] == taps) and (sets is None or got[4] == sets)
    y = torch.full((B, nz, ny, nx, cout), float("nan"), device="cuda")
    N.conv3_forward(xd, _dev(w), y)
    # three samples at most carry all the routes' edges; FP64 takes its time
    ref = np.moveaxis(U.conv3(_first(x[:3]), _w5(w)), 1, -1)
    err = np.abs(y[:3].cpu().numpy() - ref).max() / np.abs(ref).max()
    last = np.moveaxis(U.conv3(_first(x[-1:]), _w5(w)), 1, -1)
    err = max(err, np.abs(y[-1:].cpu().numpy() - last).max() / np.abs(last).max())
    assert torch.isfinite(y).all() and err < _sum_tol(27 * cin), err
