"""bench.py's FP64 roofline and traffic record (CPU): every step of the
algorithm is held against the pipe that the FP64 sweeps run it on, so that the
fraction is one of what bounds the kernel; and the traffic counters are taken
as a kernel's own only for the sources that make up its code."""
import os
import re

import pytest

import bench
from tests.conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2102_05287_gb300", "csrc")


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


def includes(name, seen=None):
    seen = set() if seen is None else seen
    if name not in seen and os.path.exists(os.path.join(CSRC, name)):
        seen.add(name)
        for inc in re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, name)).read()):
            includes(os.path.normpath(inc), seen)
    return seen


def test_traffic_hash_covers_every_source_of_the_sweeps():
    own = {n for n in includes("wcns_fp64.cu") if not n.startswith("..")}
    assert set(bench.KERNEL_SOURCES) == own


def test_traffic_hash_follows_each_source(monkeypatch, tmp_path):
    d = tmp_path / "paper_2102_05287_gb300" / "csrc"
    d.mkdir(parents=True)
    for n in bench.KERNEL_SOURCES:
        (d / n).write_bytes(open(os.path.join(CSRC, n), "rb").read())
    h = bench.kernel_source_hash()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_source_hash() == h
    for n in bench.KERNEL_SOURCES:
        text = (d / n).read_bytes()
        (d / n).write_bytes(text + b"\n")
        assert bench.kernel_source_hash() != h, n
        (d / n).write_bytes(text)
