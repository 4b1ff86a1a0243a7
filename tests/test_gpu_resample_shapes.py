"""lbm_resample over targets and channel counts that split the work in other
ways than the mean fields do: one and two cells wide, taller than they are wide,
one channel to hundreds (split over threads, in fours or one by one), sources
off a 16-byte boundary.  Each channel is bit for bit what a call for it alone
gives; short axes also against oracle.resample, with the bound of
test_gpu_resample.py: 1e-6 of the field's scale."""
import numpy as np
import pytest

import oracle.resample as R

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [((8, 8, 8), (8, 8, 8), 128), ((8, 8, 8), (4, 4, 4), 256), ((9, 5, 4), (3, 7, 2), 37), ((6, 6, 40), (1, 1, 300), 4),
         ((7, 6, 20), (2, 2, 1000), 4), ((6, 9, 5), (1, 77, 3), 5), ((33, 9, 8), (65, 3, 2), 12), ((16, 16, 16), (33, 31, 130), 8),
         ((5, 4, 3), (200, 9, 70), 64)]


@pytest.mark.parametrize("grid,out,channels", CASES)
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("off", [0, 1])
def test_shapes_match_oracle(grid, out, channels, layout, off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300 import lbm as B
    (nx, ny, nz), (mx, my, mz) = grid, out
    f = np.random.default_rng(channels + mx).normal(size=(channels, nz, ny, nx)).astype(np.float32)
    host = f if layout == 1 else np.ascontiguousarray(np.moveaxis(f, 0, -1))
    src = torch.empty(host.size + 4, device="cuda")[off:off + host.size]
    src.copy_(torch.from_numpy(host.reshape(-1)))
    n = channels * mz * my * mx
    buf = torch.full((n + 64,), float("nan"), device="cuda")
    B.lbm_resample(src, grid, channels, layout, buf, out, torch.cuda.current_stream().cuda_stream)
    got = buf.cpu().numpy()
    assert np.isnan(got[n:]).all()
    got = got[:n].reshape(channels, mz, my, mx)
    for c in range(channels):
        one = torch.full((mz, my, mx), float("nan"), device="cuda")
        B.lbm_resample(torch.from_numpy(f[c].copy()).cuda(), grid, 1, layout, one, out, torch.cuda.current_stream().cuda_stream)
        assert np.array_equal(one.cpu().numpy(), got[c]), c
    if max(grid) < 10:
        ref = R.resample(f.astype(np.float64), (mz, my, mx))
        assert np.abs(got - ref).max() / np.abs(ref).max() < 1e-6
