"""Which level's bottom runs in one thread-block cluster, when the device can place such a cluster and when it
cannot (fewer free SMs per cluster, less shared memory): the choice must fall back to a smaller bottom and at last
to the per-level kernels (-1), never to a launch that fails."""
import ctypes

import pytest

from tests.native import load


@pytest.fixture(scope="module")
def pick():
    f = load("cluster_level").pick_cluster_level
    return lambda n, nlev, robin, tb, limit: f((ctypes.c_int * 3)(*n), nlev, robin, tb, ctypes.c_longlong(limit))


@pytest.mark.parametrize("n,nlev,robin,tb,first,next_", [((128,) * 3, 6, 0, 4, 3, 4), ((64,) * 3, 5, 0, 4, 2, 3),
                                                        ((64,) * 3, 5, 0, 8, 3, -1), ((256,) * 3, 7, 1, 4, 4, 5)])
def test_falls_back_when_the_device_cannot_place_it(pick, n, nlev, robin, tb, first, next_):
    assert pick(n, nlev, robin, tb, 1 << 40) == first
    need = next(b for b in range(1 << 10, 201 << 10, 1 << 10) if pick(n, nlev, robin, tb, b) == first)
    assert pick(n, nlev, robin, tb, need - (1 << 10)) == next_   # one KB less than the first choice takes
    assert pick(n, nlev, robin, tb, -1) == -1                    # no cluster at all
