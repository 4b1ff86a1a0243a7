"""The FNO's kernels at the edges of their ranges against the FP64 oracle
(oracle/fno.py): the input gradients of the pointwise layers four cells at a
time and where that does not apply, and the tensor-core stages of the
transforms for row counts and sizes that leave tiles unfinished.  Bounds as
for the whole network: FP32 gradients 1e-4 (relative L2 per group); BF16
activations 2e-2 forward, 3e-2 and cosine 0.999 for the gradients."""
import numpy as np
import pytest

import oracle.fno as F
from test_gpu_fno import cosine, rel_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _run(nx, ny, nz, modes, width, hidden, lift_hidden, B, **kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300 import fno as G
    mz, my, mx = modes
    ocfg = F.FNOConfig(grid=(nz, ny, nx), cin=4, width=width, cout=4, modes=modes, layers=2, hidden=hidden,
                       lift_hidden=lift_hidden)
    gcfg = dict(nx=nx, ny=ny, nz=nz, cin=4, width=width, cout=4, mx=mx, my=my, mz=mz, layers=2, hidden=hidden,
                lift_hidden=lift_hidden, max_batch=B, **kw)
    r = np.random.default_rng(nx * ny * nz + hidden)
    x = r.normal(size=(B, 4, nz, ny, nx)).astype(np.float32)
    t = r.normal(size=(B, 4, nz, ny, nx)).astype(np.float32)
    m = (r.uniform(size=(B, nz, ny, nx)) < 0.6).astype(np.float32)
    p = F.init_params(ocfg, seed=3)
    for l in range(ocfg.layers):
        p[f"R{l}"] = p[f"R{l}"] * 30.0
    d = {k: (v.reshape(width, width, -1).transpose(2, 0, 1) if k.startswith("R") else v) for k, v in p.items()}
    cfg = G.make_config(**gcfg)
    net = G.FNO(**gcfg)
    net.set_params(G.flatten(cfg, d))
    y = net.forward(x)
    net.loss_grad(x, t, m)
    g = G.unflatten(cfg, net.grads())
    net.close()
    for l in range(ocfg.layers):
        g[f"R{l}"] = g[f"R{l}"].transpose(1, 2, 0).reshape(width, width, mz, 2 * my, 2 * mx)
    yr, tape = F.forward(p, x.astype(np.float64), ocfg, keep=True)
    gr = F.backward(p, tape, yr, t.astype(np.float64), m.astype(np.float64), ocfg)
    return y, yr, g, gr


@pytest.mark.parametrize("grid", [(6, 7, 6), (5, 6, 7), (8, 6, 10)])       # 252, 210 and 480 cells per sample
@pytest.mark.parametrize("hidden", [8, 128])
def test_pointwise_input_gradients(grid, hidden):
    y, yr, g, gr = _run(*grid, (2, 2, 2), 32, hidden, 32, 3, act_bf16=0, tensor_cores=0)
    worst = max(rel_l2(g[k], gr[k]) for k in gr)
    print(f"FNO {grid}, hidden {hidden}: worst gradient group {worst:.2e}")
    assert np.abs(y - yr).max() / np.abs(yr).max() < 1e-5
    assert worst < 1e-4


@pytest.mark.parametrize("ny,nz,modes,width,B", [(8, 4, (2, 4, 16), 32, 1), (24, 5, (2, 4, 16), 32, 2),
                                                 (16, 5, (2, 8, 16), 32, 3), (32, 4, (2, 4, 16), 32, 1),
                                                 (5, 5, (2, 2, 16), 3, 1), (7, 5, (2, 2, 16), 32, 3)])
def test_tensor_core_stages(ny, nz, modes, width, B):
    y, yr, g, gr = _run(128, ny, nz, modes, width, 128, 32, B, act_bf16=1, tensor_cores=int(width % 8 == 0))
    worst = max(rel_l2(g[k], gr[k]) for k in gr)
    print(f"FNO 128x{ny}x{nz}, width {width}: forward {rel_l2(y, yr):.2e}, worst gradient group {worst:.2e}")
    assert rel_l2(y, yr) < 2e-2
    for k in gr:
        assert cosine(g[k], gr[k]) > 0.999 and rel_l2(g[k], gr[k]) < 3e-2, k
