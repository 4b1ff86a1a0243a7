"""Convolution calls on buffers that start on any float: views one, two and
three floats into an allocation give the same bits as whole allocations, for
each route (halo block, shifted copies, split sums) and each direction."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [(3, 4, 8, 128, 32, 32), (2, 4, 4, 8, 64, 96), (2, 16, 16, 32, 96, 64), (8, 2, 2, 4, 128, 64)]


def _shift(t, k):
    v = torch.empty(t.numel() + 4, device="cuda", dtype=t.dtype)[k:k + t.numel()].view(t.shape)
    v.copy_(t)
    return v


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("k", [1, 2, 3])
def test_views_give_the_same_bits(case, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300 import unet as N
    B, nz, ny, nx, cin, cout = case
    g = torch.Generator(device="cuda").manual_seed(sum(case))
    x = torch.randn((B, nz, ny, nx, cin), generator=g, device="cuda")
    w = torch.randn((cout, cin, 27), generator=g, device="cuda")
    gy = torch.randn((B, nz, ny, nx, cout), generator=g, device="cuda")

    def call(f):
        y, gx, gw = f(torch.full_like(gy, float("nan"))), f(torch.full_like(x, float("nan"))), f(torch.full_like(w, float("nan")))
        N.conv3_forward(f(x), f(w), y)
        N.conv3_backward_data(f(gy), f(w), gx)
        N.conv3_backward_weights(f(x), f(gy), gw)
        return y, gx, gw

    ref, got = call(lambda t: t), call(lambda t: _shift(t, k))
    assert all(t.data_ptr() % 16 for t in got)
    assert torch.equal(ref[0], got[0]) and torch.equal(ref[1], got[1])
    # the weight gradient's parts are added atomically, in any order: twice the
    # bound of one sum (4 sqrt(K) 2^-24 of the largest)
    K = B * nx * ny * nz
    assert (ref[2] - got[2]).abs().max() <= 8 * K ** 0.5 * 2.0 ** -24 * ref[2].abs().max()
