"""The printed roofline of the FP64 forms is the FP64 pipe's (CPU)."""
import pytest

import bench

RES = {"kernels": {"sweep_x": (36.0, 3), "sweep_z": (45.0, 3), "step_begin": (0.03, 1)}, "ncell": 256 ** 3, "neq": 7,
       "grind": 0.39}


def _roof(form):
    return bench.pipe_roofline(form, bench.roofline_for(form, RES, 1.23, "measured", 6666.6, "measured"), 1.23)


@pytest.mark.parametrize("form", ["fp64", "fp64_fast"])
def test_fraction_is_the_pipes(monkeypatch, form):
    monkeypatch.setattr(bench, "read_traffic", lambda k: 0.813 if k == "fp64:sweep_z:pipe_fp64" else None)
    r = _roof(form)
    assert r["frac"] == 0.813 and abs(r["peak"] - 0.615) < 1e-4
    assert abs(r["achieved"] - r["frac"] * r["peak"]) < 1e-3
    # what the integer pipes do counts as work, not as a fraction of the FP64 pipe
    ops = 961 * 256 ** 3 / 15.0e-3 / 1e12
    assert abs(r["algorithmic_tops"] - ops) < 1e-3 and ops > r["peak"]


@pytest.mark.parametrize("form", ["fp64", "fp64_fast", "fp64_weno3", "fp64_3fluid"])
def test_no_fraction_without_a_count(monkeypatch, form):
    monkeypatch.setattr(bench, "read_traffic", lambda k: None)
    r = _roof(form)
    assert r["frac"] is None and r["achieved"] is None and r["algorithmic_tops"] > 0


def test_fp32_forms_as_they_were():
    rm = bench.roofline_for("mixed", RES, 77.5, "measured", 6666.6, "measured")
    assert bench.pipe_roofline("mixed", rm, 1.23) == rm
