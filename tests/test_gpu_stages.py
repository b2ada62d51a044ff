"""The staged kernels' stages and candidate buffers where every site is a
candidate: each block cuts (or, for a k above its room, flushes) its buffer
between tiles, and tiles begun before the cut overrun it into the run's list.
The register-fed kernel, whose blocks make room before every row, is the
reference; selections and states are equal exactly."""
import numpy as np
import pytest

from paper_0705_4371_gb300 import inputs
from tests._common import oracle_cfg, perturbed_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_0705_4371_gb300 import lbm as m
    m.load()
    return m


# the edges of what a block keeps (cut below 320, flushed from there on), the
# smallest and a k above the buffer; five tiles and more per block, so that
# refills after a marked one are reached
@pytest.mark.parametrize("k", [1, 200, 319, 320, 3000])
@pytest.mark.parametrize("prec", ["f64", "f32", "f16dev"])
def test_every_site_a_candidate(lbm, prec, k):
    w = inputs.cylinder(1030, 1603, 40, 400.0, delta=-1.0, k=k)
    f0 = perturbed_state(oracle_cfg(w), w, 3, 1e-3)
    got = {}
    for shape in (0, 4, 5, 6):
        with lbm.Lattice.from_workload(w, precision=lbm.PRECISIONS[prec]) as g:
            g.set_tile_shape(shape)
            g.set_state(f0)
            g.step(2)
            g.sync()
            got[shape] = (g.counts(2), g.selected(), g.get_state())
    assert got[0][1].size == k
    for shape in (4, 5, 6):
        for a, b in zip(got[0], got[shape]):
            assert np.array_equal(a, b), (prec, k, shape)


# few candidates, all of them in strips of one warp's sites: the warp's share of
# the room is used up while the block holds no more than it keeps, so the cut
# finds nothing to do and the next row's sites are appended right after it
@pytest.mark.parametrize("k", [64, 100])
@pytest.mark.parametrize("prec", ["f64", "f32dev"])
def test_a_cut_that_keeps_everything(lbm, prec, k):
    w = inputs.cylinder(1030, 803, 40, 400.0, delta=1e-6, k=k)
    f0 = perturbed_state(oracle_cfg(w), w, 3, 1e-5, noise=1e-4)
    kick = 1.0 + 1e-2 * inputs.uniform(4, f0.shape)
    strips = np.zeros(f0.shape[1:], bool)
    for y in range(3, 800, 5):
        x = 32 * (1 + (7 * y) % 29)
        strips[y, x:x + 31] = True
    f0 = np.where(strips, f0 * kick, f0)
    got = {}
    for shape in (0, 1, 2, 3, 4):
        with lbm.Lattice.from_workload(w, precision=lbm.PRECISIONS[prec]) as g:
            g.set_tile_shape(shape)
            g.set_state(f0)
            g.step(3)
            g.sync()
            got[shape] = (g.counts(3), g.selected(), g.get_state())
    assert got[4][1].size == k
    for shape in (0, 1, 2, 3):
        for a, b in zip(got[4], got[shape]):
            assert np.array_equal(a, b), (prec, k, shape)
