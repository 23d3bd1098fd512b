"""What bench.py rates a kernel against."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_products_of_fp32_heads_are_rated_by_the_units_they_run_on():
    import bench
    from paper_1806_03925_b200.workloads import PRESETS
    p = PRESETS["skew"]
    stats = dict(B=p.batch, nnz=3.0 * p.batch, uniq_img=2e4, uniq_emb=2e4, n_ready=100.0)
    peaks = dict(hbm_gbs=6500.0, bf16_tflops=1600.0, bf16_sustained=1380.0, source="test")
    fan = (p.d_in,) + p.hidden
    fwd = sum(2 * p.batch * a * b for a, b in zip(fan, p.hidden)) / 2                  # a launch: the mean of the two layers
    r = bench.roofline_for("f32_gemm_fwd", 0.0695, p, stats, peaks)
    assert r["bound"] == "alu" and abs(r["peak"] - 148 * 128 * 2 * 1.965e-3) < 0.1
    assert abs(r["frac"] - fwd / 0.0695e-3 / (148 * 128 * 2 * 1.965e9)) < 1e-3 and 0.4 < r["frac"] < 0.8
    r = bench.roofline_for("tc3_gemm_dx", 0.033, p, stats, peaks)
    assert r["bound"] == "tensor" and abs(r["peak"] - 230.0) < 0.1
    # the step's products: at least the time of each part on its own units
    r = bench.step_roofline(p, stats, 0.3, peaks)
    flops = r["flops_per_step"]
    least = flops / 3 / (148 * 128 * 2 * 1.965e9) + flops * 2 / 3 / 230e12
    assert r["lower_bound_ms"] >= round(least * 1e3, 4) - 2e-4 and abs(r["math_frac"] - least / 0.3e-3) < 1e-3
    assert bench.step_roofline(PRESETS["medium"], stats, 0.3, peaks)["math_peak"] == 1380.0
