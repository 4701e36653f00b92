"""What the bench makes of the captured steps' timing (kinds 0, 2 and 7)."""
import numpy as np
import pytest

import bench


def row(fluid, interior_bricks, boundary_bricks):
    r = np.zeros(10, np.int64)
    r[1], r[8], r[9] = fluid, interior_bricks, boundary_bricks
    return r


def test_interior_bricks_and_the_rest_launch():
    n, ms = np.array([4, 0, 4, 0, 0, 0, 0, 4]), np.array([8.0, 0, 2.0, 0, 0, 0, 0, 9.0])
    f = bench.finest_stream_collide(row(64 * 100 + 64 * 10 + 5, 100, 10), n, ms, 19, 1)
    brick, listed = bench.bytes_per_update(19, 1, brick=True), bench.bytes_per_update(19, 1)
    assert f["finest_kernel"] == "k_sc_interior" and f["finest_units"] == 6400 and f["finest_launches"] == 4
    assert f["finest_launch_ms"] == 2.0 and f["finest_gbs"] == pytest.approx(6400 * brick / 2e-3 / 1e9)
    # the rest launch holds both kinds of element
    assert f["finest_boundary_units"] == 640 and f["finest_list_units"] == 5
    assert f["finest_rest_gbs"] == pytest.approx((640 * brick + 5 * listed) / 0.5e-3 / 1e9)
    assert f["finest_sc"]["span_ms"] == 2.25
    assert f["finest_sc"]["bytes"] == pytest.approx(7040 * brick + 5 * listed)


def test_a_level_without_interior_bricks_is_timed_too():
    n, ms = np.array([0, 0, 4, 0, 0, 0, 0, 4]), np.array([0, 0, 2.0, 0, 0, 0, 0, 2.0])
    f = bench.finest_stream_collide(row(645, 0, 10), n, ms, 9, 0)
    nbytes = 640 * bench.bytes_per_update(9, 0, brick=True) + 5 * bench.bytes_per_update(9, 0)
    assert f["finest_kernel"] == "k_sc_rest" and f["finest_units"] == 645 and f["finest_launch_ms"] == 0.5
    assert f["finest_gbs"] == pytest.approx(nbytes / 0.5e-3 / 1e9)
    assert f["finest_sc"]["gbs"] == pytest.approx(f["finest_gbs"])


def test_nothing_timed():
    f = bench.finest_stream_collide(row(645, 0, 10), np.zeros(8, int), np.zeros(8), 9, 0)
    assert f["finest_launch_ms"] is None and f["finest_gbs"] is None and f["finest_sc"]["gbs"] is None
