"""Where calls of the small-network kernels go (csrc/kt_coop.cu coop_group): batches and intervals at
which one cell per lane was measured faster than the groups keep one cell per lane, and where
the groups were ahead they are taken.  Host compiler only."""
import ctypes

import numpy as np
import pytest

from test_coop_class import probe  # noqa: F401

TR, BE = 1, 0


def _lanes(probe, N, energy, form, scheme, ncells, steps):  # noqa: F811
    ns = N - energy
    nin = np.full(4, 2, np.int32)
    pin = np.array([[r % ns, (r + 1) % ns, -1] for r in range(4)], np.int32)
    out = np.zeros(7, np.int32)
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    assert probe.route_dt(N, energy, form, scheme, ncells, ctypes.c_double(steps), 4, p(nin), p(pin), p(out)) >= 0
    return int(out[0])


# unknowns, temperature, FP32-LU, scheme, cells, interval in first steps
LANE = [(11, 1, 1, TR, 48000, 0.1), (11, 1, 1, TR, 131072, 1.0), (11, 1, 1, TR, 262144, 3.0), (11, 1, 1, TR, 1048576, 10.0),
        (11, 1, 0, TR, 131072, 0.1), (11, 1, 0, TR, 524288, 1.0), (11, 1, 0, TR, 1048576, 3.0),
        (7, 1, 0, TR, 9700, 0.1), (7, 1, 0, BE, 9700, 1e-4), (7, 1, 0, TR, 200000, 10.0), (8, 1, 0, TR, 20000, 1000.0),
        (8, 1, 0, TR, 200000, 1000.0), (8, 1, 0, BE, 200000, 10.0), (10, 1, 0, TR, 14500, 1e-4), (10, 1, 0, TR, 50000, 10.0),
        (13, 1, 0, TR, 50000, 1e-4), (6, 0, 0, TR, 5000, 1e-4), (6, 0, 0, BE, 9700, 1e-4), (9, 0, 0, TR, 9700, 1e-4),
        (11, 0, 0, BE, 6000, 0.01), (11, 0, 0, TR, 9700, 1.0), (3, 0, 1, TR, 9800, 100.0), (14, 0, 0, TR, 20000, 100.0)]
GROUP = [(11, 1, 1, TR, 250, 1e-2), (11, 1, 1, TR, 12000, 0.1), (11, 1, 1, TR, 65536, 3.0), (11, 1, 1, TR, 65536, 1e6),
         (11, 1, 1, TR, 1048576, 100.0), (11, 1, 0, TR, 262144, 10.0), (11, 1, 0, BE, 1048576, 0.1), (3, 0, 1, TR, 9700, 0.1),
         (3, 0, 0, BE, 1000, 1e8), (7, 1, 0, TR, 5000, 0.1), (8, 1, 0, TR, 9700, 1000.0), (10, 1, 0, TR, 9700, 1e-4),
         (10, 1, 0, TR, 25000, 100.0), (13, 1, 0, TR, 14500, 1e-4), (13, 1, 0, TR, 100000, 10.0), (16, 1, 0, TR, 200000, 1e-4),
         (16, 1, 0, BE, 200000, 10.0), (9, 0, 0, TR, 5000, 1e-4), (11, 0, 0, TR, 9700, 1000.0), (14, 0, 0, TR, 9700, 1000.0)]


@pytest.mark.parametrize("call", LANE, ids=str)
def test_calls_that_groups_slow_down_keep_one_cell_per_lane(probe, call):  # noqa: F811
    assert _lanes(probe, *call) == 0


@pytest.mark.parametrize("call", GROUP, ids=str)
def test_calls_that_groups_speed_up_take_them(probe, call):  # noqa: F811
    assert _lanes(probe, *call) > 0


def test_steps_of_each_cells_own_count_as_long(probe):  # noqa: F811
    """kt_integrate_dt passes the intervals in device memory: their length is not known."""
    assert _lanes(probe, 11, 1, 1, TR, 1048576, -1.0) == 8
