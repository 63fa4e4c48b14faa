"""The benchmark's choice of a launch shape for the FP64 solver, whose workspace can exceed the free memory at the shape
that suits the mixed solver: it must fall back to one that fits instead of failing.  CPU only."""
import pytest

import bench

GIB = 1 << 30


def _f64_bytes(lanes, block):  # 32^3 x 64: 193.75 GiB for one lane of 64
    return lanes * block * 193.75 * GIB / 64


@pytest.mark.parametrize("lanes,block,free,want", [(1, 64, 166, (1, 32)), (1, 64, 200, (1, 64)), (1, 32, 166, (1, 32)),
                                                   (4, 16, 166, (2, 16)), (8, 64, 166, (1, 32)), (2, 64, 100, (1, 32)),
                                                   (1, 3, 4, (1, 1))])
def test_shape_that_fits(lanes, block, free, want):
    assert bench.shape_that_fits(_f64_bytes, lanes, block, free * GIB) == want


def test_nothing_fits():
    with pytest.raises(MemoryError):
        bench.shape_that_fits(_f64_bytes, 2, 16, GIB)

