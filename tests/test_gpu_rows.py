"""Staged rows whose boundary rules are written into the staged planes, and
the sites gathered with the rules one by one, against the oracle and against
each other: every kind of side, obstacles one site from the walls and the
edges, both wall rules, ragged grids, the probe on any kind of site."""
import numpy as np
import pytest

from oracle import core as ora
from paper_0705_4371_gb300 import inputs
from tests._common import oracle_cfg, perturbed_state, rel_err

pytestmark = pytest.mark.gpu

BB, FREE, IN, OUT, PER, COPY = (inputs.BC_BB, inputs.BC_FREESLIP, inputs.BC_INLET, inputs.BC_OUTLET,
                                inputs.BC_PERIODIC, inputs.BC_OUTLET_COPY)


@pytest.fixture(scope="module")
def lbm():
    from paper_0705_4371_gb300 import lbm as m
    m.load()
    return m


# (nx, ny, sides x0 x1 y0 y1, obstacle x0 y0 w h, wall, probe)
CASES = [
    (261, 41, (IN, OUT, FREE, FREE), (30, 1, 9, 8), 0, (29, 0)),
    (257, 40, (IN, COPY, FREE, BB), (1, 31, 7, 8), 1, (8, 39)),
    (140, 37, (BB, BB, BB, FREE), (131, 10, 5, 20), 0, (1, 0)),
    (129, 25, (IN, COPY, PER, PER), (60, 1, 70 - 6, 23), 1, (127, 24)),
    (130, 9, (PER, PER, BB, BB), (40, 3, 3, 3), 0, (129, 4)),
    (64, 70, (PER, PER, PER, PER), (5, 60, 30, 9), 1, (0, 0)),
    (384, 13, (COPY, IN, FREE, FREE), (0, 0, 0, 0), 0, (383, 12)),
    (5, 3, (IN, OUT, BB, BB), (0, 0, 0, 0), 0, (2, 1)),
    (300, 50, (OUT, COPY, BB, FREE), (126, 20, 4, 9), 1, (130, 19)),
]


def _workload(c):
    nx, ny, bc, ob, wall, probe = c
    w = inputs.cylinder(300, 80, 6, 400.0, delta=1e-6, k=5)
    w.nx, w.ny, w.bc, w.obstacle, w.wall, w.probe = nx, ny, bc, ob, wall, probe
    w.u_in = (0.05, 0.01)
    return w


@pytest.mark.parametrize("case", CASES)
def test_shapes_and_oracle_agree(lbm, case):
    w = _workload(case)
    cfg = oracle_cfg(w)
    f0 = perturbed_state(cfg, w, 7, 1e-3)
    steps = 6
    fo, log = ora.run(cfg, f0.copy(), steps)
    for prec in ("f64", "f32", "f32dev", "f16dev"):
        got = {}
        for shape in (0, 4, 5, 6):
            with lbm.Lattice.from_workload(w, precision=lbm.PRECISIONS[prec]) as g:
                g.set_tile_shape(shape)
                g.set_probe(*w.probe)
                g.set_state(f0)
                g.step(steps)
                g.sync()
                got[shape] = (g.get_state(), g.counts(steps), g.probe(steps), g.selected())
        for shape in (4, 5, 6):
            for a, b in zip(got[0], got[shape]):
                assert np.array_equal(a, b), (prec, shape)
        if prec == "f64":
            assert rel_err(got[5][0], fo) < 1e-12
            assert np.array_equal(got[5][3], log.selected[-1])


@pytest.mark.parametrize("eq", ["poly", "entropic"])
@pytest.mark.parametrize("k", [1, 7, 300, 4000])
def test_selection_by_counting_and_by_radix_agree(lbm, eq, k):
    # few candidates (ranked by counting), more than one per thread (radix
    # select) and more than the blocks keep; ties from a mirrored state
    w = _workload(CASES[0])
    w.eq = inputs.EQ_POLY if eq == "poly" else inputs.EQ_ENTROPIC
    w.k, w.obstacle = k, (0, 0, 0, 0)
    cfg = oracle_cfg(w)
    f0 = perturbed_state(cfg, w, 9, 1e-3)
    half = (w.ny + 1) // 2
    f0[:, half:] = f0[:, :w.ny - half]          # repeated rows: equal dS at distinct sites
    ds = ora.fields(cfg, f0)[1]
    for q in (0.3, 0.98, 0.999):
        w.delta = float(np.quantile(ds[np.isfinite(ds)], q))
        want = ora.select(ds.ravel(), w.delta, k)
        with lbm.Lattice.from_workload(w, precision=lbm.LB_F64) as g:
            g.set_state(f0)
            dsg = g.delta_s()
            g.step(1)
            assert np.array_equal(g.selected(), ora.select(dsg.ravel(), w.delta, k))
            assert g.selected().size == min(k, int((dsg > w.delta).sum()))
        assert want.size == min(k, int((ds > w.delta).sum()))
