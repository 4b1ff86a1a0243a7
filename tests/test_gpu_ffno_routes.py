"""The factorised surrogate's kernels over the lengths, widths and sizes that
take different routes, against the FP64 oracle (oracle/ffno.py): transforms
in registers (32, 48, 64, 96, 128; fewer modes than the kernel's) and from
tables (lengths of each remainder by four, odd ones), line counts that leave
tiles unfinished, cell counts that leave quadruples or pairs of cells
unfinished, hidden widths of one to four chunks, and networks past the tiled
kernels' limits.  Bounds as for the whole network in FP32."""
import numpy as np
import pytest

from oracle import ffno as F

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# grid (z, y, x), modes (z, y, x), width, cin, cout, hidden of the lift, layer and projection, batch, max_batch
CASES = {
    "registers": ((32, 48, 64), (16, 16, 32), 8, 4, 4, 8, 8, 16, 1, 1),
    "registers, long rows": ((3, 32, 96), (2, 9, 20), 32, 4, 4, 32, 32, 128, 2, 2),
    "registers, few modes": ((64, 3, 128), (11, 1, 32), 20, 3, 5, 20, 40, 33, 1, 3),
    "tables": ((50, 33, 20), (20, 10, 7), 12, 4, 4, 12, 12, 32, 2, 2),
    "tables, long": ((2, 6, 200), (1, 3, 60), 32, 4, 4, 32, 32, 64, 1, 1),
    "64 rows, 32 modes": ((64, 4, 64), (32, 2, 17), 8, 2, 3, 8, 8, 8, 1, 1),
    "odd cells": ((5, 7, 9), (3, 4, 5), 32, 4, 4, 32, 64, 128, 3, 3),
    "pairs of cells": ((5, 6, 9), (2, 3, 4), 3, 1, 1, 65, 128, 5, 2, 4),
    "wide lift": ((4, 4, 9), (2, 2, 4), 32, 9, 9, 100, 128, 70, 1, 1),
    "width past the tiles": ((6, 5, 8), (2, 3, 4), 40, 4, 4, 8, 8, 16, 2, 2),
    "hidden past the tiles": ((6, 5, 8), (2, 3, 4), 8, 4, 4, 8, 8, 160, 2, 2),
}


@pytest.mark.parametrize("name", list(CASES))
def test_matches_oracle(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300 import ffno as G
    grid, modes, width, cin, cout, lift, ff, hidden, B, most = CASES[name]
    cfg = F.FFNOConfig(grid=grid, cin=cin, width=width, cout=cout, modes=modes, layers=2, ff_hidden=ff, hidden=hidden,
                       lift_hidden=lift)
    nz, ny, nx = grid
    mz, my, mx = modes
    net = G.FFNO(nx=nx, ny=ny, nz=nz, cin=cin, width=width, cout=cout, mx=mx, my=my, mz=mz, layers=2, ff_hidden=ff,
                 hidden=hidden, lift_hidden=lift, max_batch=most)
    p = F.init_params(cfg, seed=4)
    net.set_params(G.flatten(net.cfg, p))
    r = np.random.default_rng(len(name))
    x = r.normal(size=(B, cin) + grid).astype(np.float32)
    t = r.normal(size=(B, cout) + grid).astype(np.float32)
    m = (r.uniform(size=(B,) + grid) < 0.7).astype(np.float32)
    y = net.forward(x)
    yr = F.forward(p, x.astype(np.float64), cfg)
    ferr = np.abs(y - yr).max() / np.abs(yr).max()
    L = net.loss_grad(x, t, m)
    Lr, gr = F.loss_and_grad(p, x.astype(np.float64), t.astype(np.float64), m.astype(np.float64), cfg)
    g = G.unflatten(net.cfg, net.grads())
    net.close()
    worst = max(np.linalg.norm((g[k] - gr[k]).ravel()) / (np.linalg.norm(gr[k].ravel()) + 1e-300) for k in g)
    print(f"FFNO {name}: forward {ferr:.2e}, loss {abs(L - Lr) / Lr:.2e}, worst gradient group {worst:.2e}")
    assert ferr < 1e-5 and abs(L - Lr) < 1e-6 * Lr and worst < 1e-4
