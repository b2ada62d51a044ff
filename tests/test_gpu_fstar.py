"""FP64 entropic quasiequilibria (Sec. 4.1 closed form, Sec. 4.2 product form) as
the device evaluates them, against extended precision: no further off, in the
root mean square over the range of velocities, than the printed formulas
evaluated in FP64 with correctly rounded operations."""
import numpy as np
import pytest

from paper_0705_4371_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_0705_4371_gb300 import lbm as m
    m.load()
    return m


def _tube(rho, u, one):
    s = np.sqrt(1 + 3 * u * u)
    return np.stack([2 * rho / (3 * one) * (2 - s), rho / (6 * one) * (2 * s - 3 * u - 1),
                     rho / (6 * one) * (3 * u - 1 + 2 * s)])


def _product(rho, ux, uy, one):
    cx, cy = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
    w = [4 * one / 9] + [one / 9] * 4 + [one / 36] * 4
    sx, sy = np.sqrt(1 + 3 * ux * ux), np.sqrt(1 + 3 * uy * uy)
    bx, by = (2 * ux + sx) / (1 - ux), (2 * uy + sy) / (1 - uy)
    base, px, py = rho * (2 - sx) * (2 - sy), {0: one, 1: bx, -1: 1 / bx}, {0: one, 1: by, -1: 1 / by}
    return np.stack([base * w[i] * px[cx[i]] * py[cy[i]] for i in range(9)])


@pytest.mark.parametrize("lattice", ["d1q3", "d2q9"])
def test_entropic_fstar_is_as_close_as_the_printed_formula(lbm, lattice):
    n = 400_000
    rho = 1.25 + 0.75 * inputs.uniform(3, (n,))
    ux, uy = 0.3 * inputs.uniform(4, (n,)), 0.3 * inputs.uniform(5, (n,))
    if lattice == "d1q3":
        w = inputs.shock_tube(n, 1e-3, 1e-3, 4, 1)
        shape, args, formula = (1, n), (rho, ux), _tube
    else:
        w = inputs.cylinder(640, 625, 8, 400.0, eq=inputs.EQ_ENTROPIC)
        w.obstacle, w.bc = (0, 0, 0, 0), (inputs.BC_PERIODIC,) * 4
        shape, args, formula = (625, 640), (rho, ux, uy), _product
    with lbm.Lattice.from_workload(w, precision=lbm.LB_F64) as g:
        g.init_equilibrium(*(a.reshape(shape) for a in args))
        got = g.get_state().reshape(-1, n)
    exact = formula(*(a.astype(np.longdouble) for a in args), np.longdouble(1))
    fp64 = formula(*args, 1.0)

    def rms(f):
        return float(np.sqrt(np.mean(((f - exact) / exact[0]) ** 2)))

    assert np.abs(got - fp64).max() < 1e-14
    assert rms(got) <= rms(fp64), (rms(got), rms(fp64))
