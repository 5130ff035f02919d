"""bench.py's FP64 roofline (CPU): every step of the
algorithm is held against the pipe that the FP64 sweeps run it on, so that the
fraction is one of what bounds the kernel."""
import pytest

import bench


def test_fraction_is_of_both_pipes():
    ops = bench.algorithmic_ops(128, 64)
    peaks = {"fp64_fma_tflops": 1.25, "fp32_fma_tflops": 75.0}
    ncell, ms = 2048 * 1024, 1.4
    r = bench.fp64_roofline(ops, peaks, ms, ncell, "k")
    flops = {s: sum(c.values()) for s, c in ops["per_step"].items()}
    assert set(bench.FP64_PIPE_STEPS) < set(flops)
    f64 = sum(flops[s] for s in bench.FP64_PIPE_STEPS)
    f32 = sum(flops.values()) - f64
    assert f32 > f64  # most flops are off the FP64 pipe
    t = f64 * ncell / 1.25e12 + f32 * ncell / 75e12
    assert r["frac"] == pytest.approx(t / (ms * 1e-3)) and r["frac"] < 1
    assert r["achieved"] / r["peak"] == pytest.approx(r["frac"])
    assert r["frac_fp64_pipe_alone"] == pytest.approx(sum(flops.values()) * ncell / 1.25e12 / (ms * 1e-3))
