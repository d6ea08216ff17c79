"""The benchmark's count of the particle order's radix passes and bytes: the
pass count follows from the F_max that is sorted."""
import numpy as np
import pytest

import bench


@pytest.mark.parametrize("steps,passes", [(0, 1), (2 ** 9 - 2, 1), (2 ** 9 - 1, 2), (2 ** 18 - 2, 2), (2 ** 18 - 1, 3),
                                          (2 ** 27 - 2, 3), (2 ** 27 - 1, 4), (2 ** 30, 4)])
def test_passes_of_a_range(steps, passes):
    hi = np.array([0x7f000000], np.uint32)
    lo = (hi - np.uint32(steps)).view(np.float32)[0]
    assert bench.fragment_passes(float(lo), float(hi.view(np.float32)[0])) == passes


def test_passes_of_collapse_times():
    assert bench.fragment_passes(0.0, 0.0) == 1
    assert bench.fragment_passes(1e-4, 3.0) == 3  # fifteen octaves
    assert bench.fragment_passes(1e-5, 3.0) == 4  # eighteen


def test_bytes():
    # F three times, counts, then 4 B in, 4 B out and 16 B through memory per further pass
    assert [bench.fragment_bytes(p) for p in (1, 2, 3, 4)] == [21, 37, 53, 69]
