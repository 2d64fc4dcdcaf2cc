"""Per-launch figures of bench.py for kernels that take several steps per launch."""
import pytest


def test_launch_figures():
    import bench
    # 1000 steps of 24 bytes a node in 84 launches of 12 steps (the last of 4): 1 ms in all
    f = bench.launch_figures(800, 24, 1000, 84, 1.0, "chunks", 6790.7)
    assert f["avg_launch_ms"] == pytest.approx(1.0 / 84)
    assert f["steps_per_launch"] == pytest.approx(1000 / 84)
    assert f["algorithmic_bytes_per_launch"] == 800 * 24
    assert f["bound"] == "arithmetic" and f["achieved"] is None and f["frac"] is None
    assert bench.launch_figures(800, 24, 1000, 84, 1.0, "block", 6790.7)["achieved"] is None


def test_traffic_bound_launch_figures():
    import bench
    f = bench.launch_figures(1_000_000, 36, 100, 100, 1.0, "smem_deep", 6000.0)
    assert f["bound"] == "hbm" and f["steps_per_launch"] == 1.0
    assert f["achieved"] == pytest.approx(1e6 * 36 / 1e-5 / 1e9)
    assert f["frac"] == pytest.approx(f["achieved"] / 6000.0)
