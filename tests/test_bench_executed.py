"""bench.py's FP64 roofline: beside the method's operations, those that are executed with A p kept
between the passes -- 18 operations and 80 bytes per cell and iteration, 12 and 24 per cell
and initial residual -- and the fractions from the same time (no GPU)."""
from test_bench_host import load_bench


def test_executed_operations():
    b = load_bench()
    n, cg_it = 1000, 37
    reps = [{"iters": cg_it + b.NSTEPS, "cell_updates": (cg_it + b.NSTEPS) * n}] * 2
    r = b.fp64_roofline(reps, 1, ms_per_step=2.0, steps=3, peaks={"hbm_gbs": 1000.0}, measured_tflops=1.1)
    sec, e = 2.0e-3 * 3, r["executed"]
    tf = 2 * n * (18 * cg_it + 12 * b.NSTEPS) / sec / 1e12
    gbs = 2 * n * (80 * cg_it + 24 * b.NSTEPS) / sec / 1e9
    assert abs(e["tflops"] - tf) <= 1e-12 * tf and abs(e["frac"] - tf / 1.1) <= 1e-12
    assert abs(e["hbm_gbs"] - gbs) <= 1e-12 * gbs and abs(e["hbm_frac"] - gbs / 1000.0) <= 1e-12
    assert e["tflops"] < r["achieved"] and e["hbm_gbs"] > r["hbm_achieved_gbs"]
