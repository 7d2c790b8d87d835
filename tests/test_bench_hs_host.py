"""The hard-sphere roofline's count of loads, on the CPU: trials without weight
are not loaded and do not count."""
import numpy as np

import bench


def test_only_weighted_trials_count():
    b = np.zeros((5, 32), np.float32)
    assert bench.weighted_loads(b) == 0
    b[1, 3] = b[4, 31] = 0.5
    assert bench.weighted_loads(b) == 6
    b[:] = 1.0
    assert bench.weighted_loads(b) == 3 * b.size
