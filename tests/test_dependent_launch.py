"""Kernels launched as programmatic dependents run while their predecessor still
writes the populations they will read: the kernel sources read populations by
ordinary loads only, never through the read-only path, and promise no read-only
source.  (The claim order of the staged tiles, which no kernel writes, is the
one table read that way.)"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0705_4371_gb300", "csrc")


def test_populations_are_read_by_ordinary_loads():
    for name in ("lbm_kernels.cuh", "lbm_device.cuh", "lbm_energy.cuh", "lbm_batch_kernels.cuh"):
        code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for call in re.findall(r"__ldg\s*\(([^;]*);", code):
            assert call.lstrip().startswith("P.tile_order"), (name, call)
        assert "ld.global.nc" not in code, name
        assert not re.findall(r"const\s+\w+\s*\*\s*__restrict__", code), name
