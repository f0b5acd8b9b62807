"""The bench's count of the bound pass's bytes: a culled triangle costs its
indices and its pixel box, a kept one also its record and list entry; shared
vertices are read once."""


def test_culled_triangles_leave_no_record():
    import bench
    frame = dict(vertices=700, tiles=30, cleared_pixels=0)
    kept = bench.stage_a_bytes(triangles=1000, culled=0, **frame)
    culled = bench.stage_a_bytes(triangles=1000, culled=1000, **frame)
    assert culled == 1000 * (16 + 16) + 700 * 32 + 30 * 24
    assert kept - culled == 1000 * (96 + 4 + 8)
    assert bench.stage_a_bytes(1000, 0, 700, 30, 50) - kept == 8 * 50


def test_no_more_than_a_measured_launch_moves():
    """The 64-view frame's bound pass (5,467,339 triangle-views, 3,104,163 of
    them culled, 2.6 M vertices) moved 262.7 MB in and 545.5 MB out by the
    hardware's counters, half-planes included."""
    import bench
    assert 0.5 * 808e6 < bench.stage_a_bytes(5_467_339, 3_104_163, 2_600_000, 0, 0) < 808e6
