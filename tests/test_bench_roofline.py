"""The benchmark's roofline figures from a run's kernel statistics."""
import pytest

import bench


def _plans(n, resident, steps=20000, cells=46_080_000):
    o = {"steps_per_launch": 3, "march_rows": 32, "kernel_3d": 3}
    return [(dict(o, resident=1) if resident else o, {"n_cells": cells, "launches": -(-steps // 3)}) for _ in range(n)]


@pytest.fixture(autouse=True)
def captured(monkeypatch):
    monkeypatch.setattr(bench, "traffic_per_cell", lambda kernel: (21.0, {"kernel": kernel}))


def test_resident_shapes_of_a_chunk_are_one_launch():
    # eight shapes, 108 chunks of each a step, 20 steps of 11.6 s: 108 passes over 368.6 M cells a step, 21 B a cell each
    step_ms = 20 * 11616.0
    r = bench.roofline(_plans(8, True), 20, 20 * 8 * 108, step_ms, 20 * 20000 * 368_640_000, 25, 6790.0, "measured")
    assert r["shapes_per_launch"] == 8 and r["cells_per_launch"] == 368_640_000
    assert r["avg_launch_ms"] == pytest.approx(11616.0 / 108)
    assert r["dram_gbs"] == pytest.approx(21.0 * 368_640_000 * 108 / 11.616 / 1e9)
    assert r["dram_frac"] < 0.02 and r["bound"] != "hbm"
    assert r["achieved"] == pytest.approx(25 * 20000 * 368_640_000 / 11.616 / 1e9)


def test_one_shape_for_all_plans():
    r = bench.roofline(_plans(3, True), 2, 2 * 106, 100.0, 10 ** 9, 25, 6790.0, "measured")
    assert r["shapes_per_launch"] == 1 and r["avg_launch_ms"] == pytest.approx(50.0 / 106)


def test_multi_step_kernels_launch_once_per_index():
    r = bench.roofline(_plans(8, False), 20, 20 * 6667, 20 * 14000.0, 20 * 20000 * 368_640_000, 25, 6790.0, "measured")
    assert r["kernel"].startswith("k_step2d_tk") and r["bound"] == "hbm" and r["shapes_per_launch"] == 1
    assert r["avg_launch_ms"] == pytest.approx(14000.0 / 6667)
