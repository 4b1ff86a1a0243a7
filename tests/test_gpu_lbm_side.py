"""Steps whose edge kernel runs beside the bulk kernel on a stream of its own give
the bits of the same steps one kernel after the other (a timed lattice keeps that
order): every storage, every pair of x faces, averages, snapshots, forces and wall
distances; and steps captured into a graph replay to the same bits, whether the
second stream existed before the capture or not."""
import numpy as np
import pytest

from paper_2606_16765_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GRID = (40, 14, 11)
PRIMS = [I.Primitive("sphere", (12.0, 6.3, 5.1), (5.5,))]
FACES = [("inlet", "outflow", "wall", "wall"), ("inlet", "outlet", "wall", "periodic"),
         ("periodic", "periodic", "periodic", "periodic")]


def _lattice(storage, faces, links=True):
    from paper_2606_16765_gb300.lbm import Solver
    mask = I.voxelize(GRID, PRIMS)
    s = Solver(GRID, mask, storage=storage, omega1=1.8, u_in=0.05, faces=faces, force_every=1, mean_start=2,
               mean_end=1 << 30, mean_every=3, snap_first=4, snap_every=4, snap_count=2)
    if links:
        s.set_wall_distances(I.link_wall_distances(GRID, PRIMS, mask))
    s.init_noise(9, 1e-3)
    return s


def _state(s):
    s.sync()
    return [s.pdfs(), s.mean()[0], s.snapshot(0), s.snapshot(1), s.forces()]


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s", "bf16s", "f16c"])
@pytest.mark.parametrize("faces", FACES)
def test_side_by_side_is_one_after_the_other(storage, faces):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    a, b = _lattice(storage, faces), _lattice(storage, faces)
    b.timing(True)
    for n in (1, 6, 7):                                  # odd and even first steps
        a.step(n)
        b.step(n)
    for x, y in zip(_state(a), _state(b)):
        assert np.array_equal(np.asarray(x), np.asarray(y), equal_nan=True)
    a.close()
    b.close()


@pytest.mark.parametrize("warm", [0, 2])
@pytest.mark.parametrize("storage", ["f32", "f16c"])
def test_captured_steps_replay(storage, warm):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300.lbm import Solver
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        mask = I.voxelize(GRID, PRIMS)
        make = lambda: Solver(GRID, mask, storage=storage, omega1=1.8, u_in=0.05, faces=FACES[0])  # noqa: E731
        a, b = make(), make()
        a.init_noise(9, 1e-3)
        b.init_noise(9, 1e-3)
        a.step(warm + 6)
        b.step(warm)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            b.step(2)                                    # recorded, not run: the lattice's time moves on
        for _ in range(3):
            g.replay()
        s.synchronize()
        a.sync()
        fa, fb = a.pdfs(), b.pdfs()
        a.close()
        b.close()
    assert np.array_equal(fa, fb)
