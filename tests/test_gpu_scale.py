"""FP64 storage at densities far from 1.  The method is linear in the density:
a state and a delta multiplied by a power of two give the same Ehrenfests' sites
and the same populations times that power, bit for bit, whatever the range of
the arithmetic that decides which sites need their exact dS."""
import numpy as np
import pytest

from oracle import core as ora
from paper_0705_4371_gb300 import inputs
from tests._common import oracle_cfg, perturbed_state

pytestmark = pytest.mark.gpu

BB, PER, FREE = inputs.BC_BB, inputs.BC_PERIODIC, inputs.BC_FREESLIP


@pytest.fixture(scope="module")
def lbm():
    from paper_0705_4371_gb300 import lbm as m
    m.load()
    return m


def _run(lbm, w, f0, scale, delta, shape, steps):
    w.delta = delta * scale
    with lbm.Lattice.from_workload(w, precision=lbm.LB_F64) as g:
        if shape is not None:
            g.set_tile_shape(shape)
        g.set_state(f0 * scale)
        g.step(steps)
        g.sync()
        return g.counts(steps), np.sort(g.selected()), g.get_state() / scale


@pytest.mark.parametrize("eq", [inputs.EQ_POLY, inputs.EQ_ENTROPIC])
@pytest.mark.parametrize("lattice, shape", [("d1q3", None), ("d2q9", 1), ("d2q9", 4)])
def test_selection_does_not_depend_on_the_scale_of_the_density(lbm, lattice, shape, eq):
    steps = 5
    if lattice == "d1q3":
        w = inputs.shock_tube(700, 1e-3, 1e-3, 9, 10, eq)
        cfg = oracle_cfg(w)
        f0 = ora.init_field(cfg, *inputs.shock_tube_fields(w)) * (1 + 1e-3 * inputs.uniform(5, (3, 1, 700)))
    else:
        w = inputs.cylinder(203, 61, 8, 400.0, delta=1e-6, k=9)
        w.eq, w.bc = eq, (PER, PER, FREE, BB)
        cfg = oracle_cfg(w)
        f0 = perturbed_state(cfg, w, 11, 1e-3)
    ds = ora.fields(cfg, f0)[1]
    ds = ds[np.isfinite(ds)]                     # (NaN inside the obstacle)
    # half of the sites, a handful of them, and every site off equilibrium
    for delta in (float(np.median(ds[ds > 0])), float(np.quantile(ds, 0.995)), 0.0):
        want = _run(lbm, w, f0, 1.0, delta, shape, steps)
        assert want[0].sum() > 0
        for e in (-300, -90, -60, 60, 90, 300):
            got = _run(lbm, w, f0, 2.0 ** e, delta, shape, steps)
            for a, b in zip(want, got):
                assert np.array_equal(a, b), (delta, e)
