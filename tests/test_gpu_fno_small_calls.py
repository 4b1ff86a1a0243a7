"""The FNO's forward gives a sample the same bits alone as in a batch: few rows
and lines are spread over the chip in other portions than many (one or two
m-tiles per pass of the x stage, one to twelve line warps per block of the layer
kernel), without a change in any sum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ny,nz,batch", [(5, 3, 2), (8, 8, 48), (16, 16, 8), (24, 40, 3)])
def test_alone_as_in_a_batch(ny, nz, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300.fno import FNO
    net = FNO(nx=128, ny=ny, nz=nz, mx=16, my=2, mz=1, layers=2, max_batch=batch)
    x = torch.randn((batch, 4, nz, ny, 128), generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    y = net.forward(x, torch.full_like(x, float("nan"))).clone()
    for b in range(batch):
        one = net.forward(x[b:b + 1].contiguous(), torch.full_like(x[:1], float("nan")))
        assert torch.equal(one[0], y[b]), b
    net.close()
    assert torch.isfinite(y).all()
