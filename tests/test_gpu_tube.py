"""Short D1Q3 runs (many steps per cluster launch) against one launch per step
(timing mode) and against the oracle: block edges, every kind of end, sites
of one block, the largest clustered and the smallest unclustered run, selections
of each kind (all candidates, by counting, by radix)."""
import numpy as np
import pytest

from oracle import core as ora
from paper_0705_4371_gb300 import inputs
from tests._common import oracle_cfg, rel_err

pytestmark = pytest.mark.gpu

BB, IN, OUT, PER, COPY = (inputs.BC_BB, inputs.BC_INLET, inputs.BC_OUTLET, inputs.BC_PERIODIC, inputs.BC_OUTLET_COPY)


@pytest.fixture(scope="module")
def lbm():
    from paper_0705_4371_gb300 import lbm as m
    m.load()
    return m


def _run(lbm, w, prec, f0, steps, single, collision=0):
    with lbm.Lattice.from_workload(w, precision=lbm.PRECISIONS[prec]) as g:
        g.set_collision(collision)
        g.set_probe(min(w.nx - 1, 17), 0)
        g.set_timing(single)
        g.set_state(f0)
        for n in steps:
            g.step(n)
        g.sync()
        n = sum(steps)
        return g.get_state(), g.counts(n), g.probe(n), g.selected()


@pytest.mark.parametrize("n, ends, k, delta, eq", [
    (3, (BB, BB), 2, 1e-9, inputs.EQ_POLY), (16, (PER, PER), 4, 1e-8, inputs.EQ_ENTROPIC),
    (17, (IN, OUT), 3, 1e-8, inputs.EQ_POLY), (500, (IN, COPY), 4, 1e-5, inputs.EQ_ENTROPIC),
    (801, (BB, BB), 0, 1e-3, inputs.EQ_ENTROPIC), (800, (BB, BB), 300, -1.0, inputs.EQ_ENTROPIC),
    (1000, (PER, PER), 30, 1e-9, inputs.EQ_POLY), (4096, (BB, BB), 4, 1e-6, inputs.EQ_ENTROPIC),
    (4097, (BB, OUT), 4, 1e-6, inputs.EQ_ENTROPIC)])
def test_cluster_steps_equal_single_steps(lbm, n, ends, k, delta, eq):
    w = inputs.shock_tube(n, 1e-3, delta, k, 10, eq)
    w.bc = ends + (BB, BB)
    w.u_in = (0.03, 0.0)
    cfg = oracle_cfg(w)
    rho, ux, uy = inputs.shock_tube_fields(w)
    f0 = ora.init_field(cfg, rho, ux, uy) * (1 + 1e-3 * inputs.uniform(5, (3, 1, n)))
    for prec in ("f64", "f32", "f32dev", "f16dev"):
        a = _run(lbm, w, prec, f0, (7, 1, 4), False)
        b = _run(lbm, w, prec, f0, (12,), True)
        for u, v in zip(a, b):
            assert np.array_equal(u, v), prec
    fo, log = ora.run(cfg, f0.copy(), 12)
    a = _run(lbm, w, "f64", f0, (12,), False)
    if delta > 0:
        assert rel_err(a[0], fo) < 1e-12
        assert np.array_equal(a[3], log.selected[-1])


def test_elbm_tube_equals_single_steps(lbm):
    w = inputs.shock_tube(800, 1e-9, 1e-4, 4, 10)
    cfg = oracle_cfg(w)
    f0 = ora.init_field(cfg, *inputs.shock_tube_fields(w))
    a = _run(lbm, w, "f64", f0, (40,), False, lbm.LB_COLLISION_ELBM)
    b = _run(lbm, w, "f64", f0, (40,), True, lbm.LB_COLLISION_ELBM)
    for u, v in zip(a, b):
        assert np.array_equal(u, v)


def test_more_steps_than_a_launch_and_than_the_logs_hold(lbm):
    # launches of 4096 steps, and logs that wrap after 65 536: the tail of the
    # run in single steps gives the same state, counts and probe series
    w = inputs.shock_tube(100, 1.0 / 30.0, 1e-9, 3, 10)
    cfg = oracle_cfg(w)
    f0 = ora.init_field(cfg, *inputs.shock_tube_fields(w)) * (1 + 1e-3 * inputs.uniform(5, (3, 1, 100)))
    total, single, log = 66_001, 700, 65_536

    def run(parts):
        with lbm.Lattice.from_workload(w, precision=lbm.LB_F64) as g:
            g.set_probe(17, 0)
            g.set_state(f0)
            for n, timed in parts:
                g.set_timing(timed)
                g.step(n)
            g.sync()
            return g.get_state(), g.counts(log), g.probe(log), g.selected()

    want = run([(total - single, False), (single, True)])
    for parts in ([(total, False)], [(5000, False), (1, False), (total - 5001, False)]):
        for u, v in zip(run(parts), want):
            assert np.array_equal(u, v)
    for u, v in zip(_run(lbm, w, "f64", f0, (4097,), False), _run(lbm, w, "f64", f0, (4097,), True)):
        assert np.array_equal(u, v)
