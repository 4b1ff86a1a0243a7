"""A lattice on a stream of its own while the default stream is busy: wall
distances, probes and a checkpoint's state set between steps are there for the
next step (bit for bit the run with an idle default stream)."""
import numpy as np
import pytest

from paper_2606_16765_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _run(tmp_path, busy):
    from paper_2606_16765_gb300.lbm import Solver
    grid = (24, 12, 12)
    prims = [I.Primitive("sphere", (7.0, 5.5, 5.5), (5.0,))]
    mask = I.voxelize(grid, prims)
    links = I.link_wall_distances(grid, prims, mask)
    with torch.cuda.stream(torch.cuda.Stream()):
        s = Solver(grid, mask, storage="f32", omega1=1.8, u_in=0.05, force_every=1)
        s.step(4)
        s.save(str(tmp_path / "a"))
        s.step(3)
        busy()
        s.load(str(tmp_path / "a"))
        s.set_probes(np.array([3, 500, 900]))
        s.set_wall_distances(links)
        s.step(6)
        s.sync()
        out = s.pdfs(), s.probes(), s.forces()
        s.close()
    return out


def test_uploads_are_ordered_on_the_lattices_stream(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ref = _run(tmp_path, lambda: None)
    got = _run(tmp_path, lambda: torch.cuda._sleep(200_000_000))
    for a, b in zip(ref, got):
        assert np.array_equal(np.asarray(a), np.asarray(b), equal_nan=True)
