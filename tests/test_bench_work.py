"""Roofline arithmetic of the bench by the arithmetic that ran (no GPU)."""
import bench


def test_operations_over_the_units_that_run_them():
    w = [{"flops_fp64": 1e12, "flops_two_float": 2e12, "flops_fp32": 0.5e12},
         {"flops_fp64": 0.0, "flops_two_float": 2e12, "flops_fp32": 0.5e12}]
    st = bench.pipe_work(w)
    assert st == {"flops_model": 6e12, "flops_model_fp32": 1e12, "flops_two_float": 4e12}
    r = bench.mixed_peak_frac(st, 2000.0)
    assert r["fp64_achieved_tflops"] == 0.5 and r["two_float_achieved_tflops"] == 2.0
    assert r["fp32_achieved_tflops"] == 0.5
    assert abs(r["two_float_frac"] - 20.0 / bench.FP32_PEAK_TFLOPS) < 1e-12
    assert abs(r["combined"] - (r["fp64_frac"] + r["two_float_frac"] + r["fp32_frac"])) < 1e-12
    s = bench.work_shares(st)
    assert abs(s["two_float_flop_share"] - 2 / 3) < 1e-12 and abs(s["fp32_flop_share"] - 1 / 6) < 1e-12
