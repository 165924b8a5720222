"""Algorithmic work of the dominant kernel where the stage update is a kernel of its own (CPU)."""
import bench


def test_split_update_is_not_counted_to_the_last_sweep():
    kernels = {"sweep_x": (9.0, 9), "sweep_y": (8.0, 9), "sweep_z": (12.0, 9), "stage_update": (3.0, 9), "step_begin": (0.03, 3)}
    res = {"kernels": kernels, "ncell": 256 ** 3, "neq": 7, "grind": 0.02}
    r = bench.roofline_for("gated", res, 77.5, "measured", 6666.6, "measured")
    assert r["kernel"] == "sweep_z" and abs(r["avg_launch_ms"] - 12.0 / 9) < 1e-4
    assert r["algorithmic_flops_per_cell"] == bench.flops_cell_dir() + 7   # accumulation only
    whole = dict(res, kernels=dict(kernels, stage_update=(0.0, 0)))
    r = bench.roofline_for("gated", whole, 77.5, "measured", 6666.6, "measured")
    assert r["algorithmic_flops_per_cell"] == bench.flops_cell_dir() + bench.flops_last_sweep_extra()
