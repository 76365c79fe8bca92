"""Device memory of a batched lattice.

A batch never takes many steps of a lattice in one launch, so its lattices hold
no state for that, and the footprint that the server admits by has none: the same
for a lattice that would be stepped so by itself and for one that would not.
"""
import pytest

from paper_0704_0043_gb300 import lbm

SMALL = dict(lattice=lbm.D2Q9, nx=64, ny=64, precision=lbm.FP32, limiters=lbm.LIM_MEDIAN)


def test_footprint_is_that_of_a_step_a_launch():
    assert lbm.footprint_bytes(**SMALL) == lbm.footprint_bytes(kernel=lbm.KERNEL_TILED, **SMALL)


@pytest.mark.gpu
def test_batched_lattice_takes_its_footprint():
    b = lbm.Batch()
    b.add(**SMALL)
    assert b.device_bytes() == lbm.footprint_bytes(**SMALL)  # no tables before the first step
    alone, other = lbm.Lattice(**SMALL), lbm.Lattice(kernel=lbm.KERNEL_TILED, **SMALL)
    assert 0 < alone.device_bytes() - other.device_bytes() <= 32768
