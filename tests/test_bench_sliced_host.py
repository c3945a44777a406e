"""bench.py's rating of FP64-class H.X that ran as slice products (no GPU): classes of their own
against the digit products' rate on the tensor cores, not the FP64 or FP32 pipe they do not use."""
import math

import pytest

import bench
import workloads as W
from tests.test_bench_host import _FakeLib, _profile


def test_slice_products_are_rated_against_the_digit_products():
    pytest.importorskip("torch")
    from paper_1404_3773_gb300 import CS_DF64, CS_FP64, CS_MIXED_BF16

    w = W.erf_cluster_32()
    # ten iterations: a double-float Rayleigh-Ritz H.X of 1.49 ms that ran as slice products
    ms, n = _profile({"dense": (13.0, 180), "angular_f32": (28.2, 160),
                      "radial_synth_df64": (1.7, 10), "angular_df64": (11.4, 10),
                      "radial_anal_df64": (1.8, 10)})
    zero_ms, zero_n = _profile({})
    s_ms, s_n = _profile({"radial_synth_df64": (1.7, 10), "angular_df64": (11.4, 10),
                          "radial_anal_df64": (1.8, 10)})
    _, classes = bench.roofline_table(_FakeLib, w, 46128, 80, CS_MIXED_BF16, ms, n, 10, CS_DF64,
                                      (s_ms, s_n))
    assert set(classes) == {"dense", "angular_f32", "radial_synth_sliced", "angular_sliced",
                            "radial_anal_sliced"}
    c = classes["angular_sliced"]
    assert c["launches"] == 10 and c["bound"] == "tensor"
    peak = bench.measured_peaks()["bf16_tflops_sustained"] / 34.0
    assert c["peak"] == round(peak, 3)
    ach = bench.algorithmic_flops(w, 80)["angular"] / 1.14e-3 / 1e12
    assert math.isclose(c["achieved"], ach, rel_tol=1e-3)
    # against the FP64 pipe the same class would read 2.5 / 1.25 TFLOP/s
    assert ach > bench.FP64_PEAK_TFLOPS
    assert all(x["frac"] is None or x["frac"] <= 1.0 for x in classes.values())
    t = bench.step_breakdown(classes, 10, 16, 9.0, CS_MIXED_BF16, CS_DF64)
    assert math.isclose(t["rayleigh_ritz_apply_ms"], 1.49, rel_tol=1e-3)
    assert math.isclose(t["filter_pass_ms"], 2.82, rel_tol=1e-3)

    # FP64 filter and Rayleigh-Ritz share the slice-product classes; without any nothing changes
    ms, n = _profile({"radial_synth": (30.0, 170), "angular": (200.0, 170),
                      "radial_anal": (25.0, 170)})
    _, classes = bench.roofline_table(_FakeLib, w, 46128, 80, CS_FP64, ms, n, 10, CS_FP64, (ms, n))
    t = bench.step_breakdown(classes, 10, 16, 26.0, CS_FP64, CS_FP64)
    assert math.isclose(t["rayleigh_ritz_apply_ms"], 1.5, rel_tol=1e-3)
    assert math.isclose(t["filter_pass_ms"], 24.0, rel_tol=1e-3)
    a = bench.roofline_table(_FakeLib, w, 46128, 80, CS_FP64, ms, n, 10, CS_FP64)
    b = bench.roofline_table(_FakeLib, w, 46128, 80, CS_FP64, ms, n, 10, CS_FP64, (zero_ms, zero_n))
    assert a == b and set(a[1]) == {"radial_synth", "angular", "radial_anal"}
