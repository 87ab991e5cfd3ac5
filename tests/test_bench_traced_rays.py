"""bench.py credits the forward trace with the rays it traces: every ray off the sensor's x axis, on it
those of the pupil rows up to the middle one (all of them at n = 2 m come in pairs, an odd grid has a
middle row of its own)."""
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402
import workloads as W  # noqa: E402


def count(n, mirrored):
    rows = [sum((2 * i + 1 - n) ** 2 + (2 * j + 1 - n) ** 2 <= n * n for i in range(n))
            for j in range(n)]
    return sum(rows[:n // 2]) + (rows[n // 2] if n % 2 else 0) if mirrored else sum(rows)


def test_traced_rays():
    reqs = np.zeros(7, dtype=W.REQ_DTYPE)
    reqs["n_grid"] = [2, 3, 64, 64, 97, 97, 33]
    reqs["v_mm"] = [0.0, 0.0, 0.0, 0.5, -0.1, 0.0, 0.0]
    want = sum(count(int(n), v == 0) for n, v in zip(reqs["n_grid"], reqs["v_mm"]))
    assert bench.traced_rays(reqs) == want
    even = reqs[2:3]
    assert 2 * bench.traced_rays(even) == bench.in_pupil_rays(64) == count(64, False)
