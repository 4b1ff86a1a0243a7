"""A network created on a stream of its own, while the default stream is busy,
starts from the parameters that it reports: its first result is bit for bit
the one after those parameters are set again."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _ffno():
    from paper_2606_16765_gb300.ffno import FFNO
    return FFNO(nx=16, ny=8, nz=8, cin=2, width=8, cout=2, mx=4, my=3, mz=3, layers=2, ff_hidden=8, hidden=16,
                lift_hidden=8, max_batch=1), (1, 2, 8, 8, 16)


def _fno():
    from paper_2606_16765_gb300.fno import FNO
    return FNO(nx=16, ny=8, nz=8, cin=2, width=8, cout=2, mx=4, my=3, mz=3, layers=2, hidden=16, lift_hidden=8,
               max_batch=1), (1, 2, 8, 8, 16)


def _unet():
    from paper_2606_16765_gb300.unet import UNet
    return UNet(nx=16, ny=8, nz=8, cin=2, cout=2, stages=1, channels=[32], bottleneck=32, max_batch=1), (1, 2, 8, 8, 16)


@pytest.mark.parametrize("make", [_ffno, _fno, _unet])
@pytest.mark.parametrize("busy", [0, 200_000_000])       # about a tenth of a second
def test_first_result_is_that_of_the_parameters(make, busy):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    make()[0].close()                                    # library loaded, kernels too
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    if busy:
        torch.cuda._sleep(busy)
    with torch.cuda.stream(s):
        net, shape = make()
        x = np.random.default_rng(1).normal(size=shape).astype(np.float32)
        first = net.forward(x)
        net.set_params(net.params())
        again = net.forward(x)
        net.close()
    assert np.array_equal(first, again)
