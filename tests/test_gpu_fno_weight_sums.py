"""Weight gradients summed over millions of cells on tensor cores, in a case
whose sums are known exactly.

With all weights zero but the last layer's bias (8, where GELU is the identity)
and the output row of channel 0 (1/2), the projection sees v = 8 everywhere, its
sine is at 0 (slope omega0 = 32, exactly) and the output is 0.  The gradient at
its 128 hidden units is then -t/(4 B N) * 2 * 1/2 * 32 with t the targets, whole
numbers below 2^16 (a BF16 pair each) and B N a power of two: every product is
exact, and so is its sum in whole numbers.

Bound: the tensor cores drop what lies below the accumulator's last place, half
a unit of 2^-23 on average, while the accumulator grows to its final value (half
of it on average).  128 products a fragment (64 steps, high and low parts) lose
128 * 2^-24 * 1/2 = 2^-18 of the sum; the sums of the fragments round to nearest
(132 of them, 2^-24 sqrt(132) / 2 < 2^-21)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("batch,hidden", [(8, 128), (8, 32), (1, 128)])
def test_long_sums(batch, hidden):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300 import fno as G
    nx, ny, nz = 128, 64, 64
    net = G.FNO(nx=nx, ny=ny, nz=nz, mx=2, my=2, mz=2, layers=1, hidden=hidden, omega0=32.0, max_batch=batch)
    d = G.unflatten(net.cfg, np.zeros(net.num_params, np.float32))
    d["W0_b"][:] = 8.0
    d["Q2_w"][0, :] = 0.5
    net.set_params(G.flatten(net.cfg, d))
    g = torch.Generator(device="cuda").manual_seed(5)
    k = torch.randint(1, 1 << 16, (batch, 1, nz, ny, nx), generator=g, device="cuda")
    t = torch.zeros((batch, 4, nz, ny, nx), device="cuda")
    t[:, :1] = k.float()
    net.loss_grad(torch.zeros_like(t), t, torch.ones((batch, nz, ny, nx), device="cuda"))
    gr = G.unflatten(net.cfg, net.grads())
    net.close()
    exact = -32.0 * int(k.sum().item()) / (4 * batch * nx * ny * nz)
    eb, ew = np.abs(gr["Q1_b"] / exact - 1).max(), np.abs(gr["Q1_w"] / (8 * exact) - 1).max()
    print(f"batch {batch}, {hidden} outputs: bias {eb:.2e}, weights {ew:.2e}")
    assert max(eb, ew) < 2.0 ** -18 + 2.0 ** -21
