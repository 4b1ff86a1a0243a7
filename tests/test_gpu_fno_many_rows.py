"""The FNO's y stages for grids with many rows and y modes: twiddle fragments
past the 48 KB that a kernel has without asking (128 rows, 32 modes), past
100 KB (192 rows, 40 modes), and past what the tensor-core kernel takes at all
(128 rows, 128 modes: the general stages).  Bounds as in test_gpu_fno_routes.py."""
import pytest

from test_gpu_fno import cosine, rel_l2
from test_gpu_fno_routes import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,my", [(128, 16), (192, 20), (128, 64)])
def test_many_rows(ny, my):
    y, yr, g, gr = _run(128, ny, 4, (1, my, 16), 8, 16, 8, 1, act_bf16=1, tensor_cores=1)
    worst = max(rel_l2(g[k], gr[k]) for k in gr)
    print(f"FNO 128x{ny}x4, {my} y modes: forward {rel_l2(y, yr):.2e}, worst gradient group {worst:.2e}")
    assert rel_l2(y, yr) < 2e-2
    for k in gr:
        assert cosine(g[k], gr[k]) > 0.999 and rel_l2(g[k], gr[k]) < 3e-2, k
