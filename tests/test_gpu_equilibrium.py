"""lbm_init_equilibrium near rest and far from it, read back through lbm_read_macros.

The momentum of the product-form equilibrium is rho u exactly.  Each stored
deviation f_i - w_i is off by its rounding r_i = eps |f_i - w_i| + tiny at most
(half a unit of the storage's last place, half a step of its smallest numbers),
so component a of the velocity is off by no more than
sum_i (|c_ia| + |u_a|) r_i / rho.  The bound carries 1.001 for the second-order
terms of that estimate and of the arithmetic before the rounding.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# storage: half a unit of the last place (relative), half a step of the subnormals
ROUND = {"f64": (2.0 ** -53, 0.0), "f32": (2.0 ** -24, 2.0 ** -150), "f16s": (2.0 ** -11, 2.0 ** -25),
         "f16c": (2.0 ** -12, 2.0 ** -26)}
C = [(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1) for i in range(27)]


def _deviations(u, p):
    """f_i - w_i in extended precision, from the small terms (no cancellation)."""
    u, p = u.astype(np.longdouble), p.astype(np.longdouble)
    third = np.longdouble(1) / 3
    out = []
    for c in C:
        e, base = 3 * p, np.longdouble(1)
        for a in range(3):
            t = 2 * third if c[a] == 0 else third / 2
            d = -u[..., a] ** 2 if c[a] == 0 else (u[..., a] ** 2 + c[a] * u[..., a]) / 2
            e, base = e * (t + d) + base * d, base * t
        out.append(e)
    return np.array(out)


@pytest.mark.parametrize("storage,scale", [("f32", v) for v in (15.9, 0.08, 1e-4, 1e-7, 1e-9, 1e-12, 1e-20)] +
                         [(s, v) for s in ("f16s", "f16c") for v in (0.08, 1e-2, 1e-4)] +
                         [("f32", 40.0), ("f64", 0.08), ("f64", 40.0)])
def test_velocity_is_exact_to_the_storage(storage, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300.lbm import Solver
    g = (13, 7, 5)
    r = np.random.default_rng(7)
    fields = (scale * r.uniform(-1, 1, (5, 7, 13, 4)) * np.array([1, 1, 1, 0.01])).astype(np.float32)
    fields[0, 0, :, 1] = -fields[0, 0, :, 0]             # linear terms that cancel
    fields[1, 0, :, 3] = 0
    s = Solver(g, None, storage=storage, omega1=1.5)
    s.init_equilibrium(fields)
    rho, u = s.macros()
    s.close()
    dev = np.abs(_deviations(fields[..., :3], fields[..., 3])).astype(np.float64)
    eps, tiny = ROUND[storage]
    if storage == "f64":
        dev = dev + 1                                    # its arithmetic rounds f_i, not the deviation
        eps *= 16                                        # a dozen operations of half a unit each
    for a in range(3):
        ua = fields[..., a].astype(np.float64)
        bound = 1.001 * sum((abs(c[a]) + np.abs(ua)) * (eps * dev[i] + tiny) for i, c in enumerate(C)) / np.abs(rho)
        err = np.abs(u[..., a] - ua)
        print(f"{storage} {scale:g} axis {a}: worst error over bound {(err / bound).max():.3f}")
        assert (err <= bound).all()


@pytest.mark.parametrize("storage", ["f32", "bf16s", "f16s", "f16c"])
def test_a_cell_that_is_not_a_number_spoils_no_other(storage):
    """Cells outside the paired arithmetic's range keep to themselves (F16C has
    no NaN: its largest code)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_16765_gb300.lbm import Solver
    g = (9, 4, 3)
    fields = np.random.default_rng(8).uniform(-0.05, 0.05, (3, 4, 9, 4)).astype(np.float32)
    a, b = Solver(g, None, storage=storage, omega1=1.5), Solver(g, None, storage=storage, omega1=1.5)
    a.init_equilibrium(fields)
    odd = fields.copy()
    odd[1, 2, 3] = np.nan
    odd[1, 2, 5, 0] = np.inf
    b.init_equilibrium(odd)
    fa, fb = a.pdfs(), b.pdfs()
    a.close()
    b.close()
    for x in (3, 5):
        if storage != "f16c":
            assert not np.isfinite(fb[:, 1, 2, x]).all()
        fb[:, 1, 2, x] = fa[:, 1, 2, x]
    assert np.array_equal(fa, fb)
