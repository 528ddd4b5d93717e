"""bench.py's roofline record where the library chooses the path (CPU)."""
import bench


def _roof():
    return {"bound": "hbm", "kernel": "k_bus", "achieved": 1500.0, "peak": 6800.0, "unit": "GB/s", "frac": 0.22,
            "traffic": None, "timing": "stamps"}


def test_fraction_of_kernels_that_the_steps_do_not_run_is_not_the_steps():
    r = bench.path_roofline(_roof(), 16, 16, 8.2)
    assert r["frac"] is None and r["kernel"] == "k_crs" and r["resident"]["us_per_iteration"] == 8.2
    assert r["per_iteration_kernels"]["frac"] == 0.22 and "do not run" in r["per_iteration_kernels"]["timing"]


def test_mixed_paths_keep_the_kernels_record():
    r = bench.path_roofline(_roof(), 48, 64, 70.0)
    assert r["frac"] == 0.22 and r["kernel"] == "k_bus" and "48 of 64" in r["timing"]
