"""The factorised surrogate on device tensors, used where they are: whole
allocations and views on 4- and 8-byte boundaries, batches past max_batch, and
a result written over the input, against the same call on host arrays (staged
into aligned buffers).  Cells in twos and fours or one by one give the same sums
per cell; the weight gradients' blocks take the same cells in the same order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [dict(nx=16, ny=8, nz=6, mx=5, my=3, mz=2, width=32), dict(nx=9, ny=7, nz=5, mx=4, my=3, mz=2, width=12),
          dict(nx=6, ny=5, nz=3, mx=2, my=2, mz=2, width=40)]                    # the last one: general kernels


def _net(shape, most, cin=4, cout=4):
    from paper_2606_16765_gb300.ffno import FFNO
    return FFNO(cin=cin, cout=cout, layers=2, ff_hidden=shape["width"], hidden=24, lift_hidden=8, max_batch=most, **shape)


def _view(a, k):
    t = torch.empty(a.size + 4, device="cuda")[k:k + a.size].view(a.shape)
    t.copy_(torch.from_numpy(a))
    return t


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("k", [0, 1, 2, 3])
def test_views_on_any_float(shape, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    grid = (shape["nz"], shape["ny"], shape["nx"])
    r = np.random.default_rng(3)
    x, t = (r.normal(size=(5, 4) + grid).astype(np.float32) for _ in range(2))
    m = r.uniform(size=(5,) + grid).astype(np.float32)
    net = _net(shape, 2)
    ref = net.forward(x)                                   # three chunks: 2, 2 and 1 samples
    out = _view(np.full_like(t, np.nan), k)
    net.forward(_view(x, k), out)
    assert np.array_equal(out.cpu().numpy(), ref)
    both = _view(x, k)                                     # the result over the input
    net.forward(both, both)
    assert np.array_equal(both.cpu().numpy(), ref)
    host = net.loss_grad(x[:2], t[:2], m[:2]), net.grads()
    dev = net.loss_grad(_view(x[:2], k), _view(t[:2], k), _view(m[:2], k)), net.grads()
    net.close()
    assert host[0] == dev[0]
    # one and the same order of the sums per gradient; the two routes of the
    # copies differ in nothing that is computed
    assert np.array_equal(host[1], dev[1])


def test_a_captured_forward_replays():
    """Device x and y: launches only, so a forward can be captured."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = torch.cuda.Stream()
    shape = SHAPES[0]
    with torch.cuda.stream(s):
        net = _net(shape, 2)
        x = torch.randn((2, 4, shape["nz"], shape["ny"], shape["nx"]), device="cuda")
        y = torch.empty_like(x)
        ref = net.forward(x, torch.empty_like(x)).clone()
        g = torch.cuda.CUDAGraph()
        s.synchronize()
        with torch.cuda.graph(g, stream=s):
            net.forward(x, y)
        y.zero_()
        g.replay()
        s.synchronize()
        assert torch.equal(y, ref)
        x.mul_(-1)
        g.replay()
        s.synchronize()
        assert not torch.equal(y, ref)
        net.close()
