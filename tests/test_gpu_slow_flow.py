"""Slow motion in water (c about 1600 m/s): the FP64 sweeps' right-hand side
keeps the accuracy of the motion itself, not that of c, against the oracle
built in long double on the same inputs.  Root mean square of the error over
that of the field, 40 cells a wavelength n / (2 pi) = 6.4 cells a radian:
- a shear of amplitude A carried at 10 m/s: the carrying velocity's rounding
  comes from the pressure's, 2^-53 (E / Gamma) / (rho c) = 1.8e-13 m/s, or
  1.8e-14 of it: 16 roundings of that size, times 6.4, are 1.8e-12;
- a pressure wave of 1.5 Pa on 15 Pa in water at rest (no kinetic energy, E - Pi
  exact): roundings of 2^-53 of ten times the wave, 16 of them, times 6.4 and
  times ten for the weights' response to the 4e-7 Pa steps that E has there:
  1.1e-12 of the momentum's rate (the wave's first-order effect; the other
  fields' rates are the scheme's dissipation, far below their own terms)."""
import ctypes as C
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_2102_05287_gb300 import problems as P  # noqa: E402
from paper_2102_05287_gb300.wcns import Solver  # noqa: E402

EOS = P.WORKLOAD_EOS
N = 40
PER = ("periodic", "periodic")


@pytest.fixture(scope="module")
def long_oracle(tmp_path_factory):
    d = tmp_path_factory.mktemp("oracle")
    src = open(O._SRC).read()
    assert src.count("typedef double real;") == 1
    (d / "o.cpp").write_text(src.replace("typedef double real;", "typedef long double real;"))
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", str(d / "o.cpp"), "-o", str(d / "o.so")],
                   check=True)
    return C.CDLL(str(d / "o.so"))


def errors(lib, n, W, dt=1e-9):
    nd = len(n)
    o = O.Oracle(n, (0.0,) * nd, (1.0,) * nd, (PER,) * nd, **EOS)
    ref = np.empty_like(W)
    p = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))  # noqa: E731
    lib.oc_rhs(C.byref(o.cfg), p(W), p(ref), C.c_double(dt), C.byref(o.stats))
    s = Solver(n, (0.0,) * nd, (1.0,) * nd, (PER,) * nd, **EOS)
    got = s.rhs(torch.from_numpy(W).cuda(), dt).cpu().numpy()
    s.close()
    rms = lambda a: np.sqrt((a ** 2).reshape(a.shape[0], -1).mean(axis=1))  # noqa: E731
    return rms(got - ref) / np.maximum(rms(ref), 1e-300)


def wave():
    x = 2 * np.pi * (np.arange(N) + 0.5) / N
    return np.sin(x) + 0.3 * np.sin(2 * x + 0.3)


@pytest.mark.parametrize("A", [1e-9, 1e-6, 1e-3, 1.0])
@pytest.mark.parametrize("axis", [0, 1])
def test_shear(long_oracle, A, axis):
    a1, w = np.full(N, 1 - 1e-6), wave()
    vel = [10.0 + 0 * w, A * w]
    W = P.conservative(EOS, a1 * 1000, (1 - a1) * 1.0, vel if axis == 0 else vel[::-1], 1e5 + 0 * w, a1)
    W = np.repeat(W[:, None, :], 3, 1) if axis == 0 else np.repeat(W[:, :, None], 3, 2)
    e = errors(long_oracle, (N, 3) if axis == 0 else (3, N), np.ascontiguousarray(W))
    assert e[3 - axis] <= 1.8e-12, e


def test_pressure_wave_at_rest(long_oracle):
    a1, w = np.full(N, 1 - 1e-6), wave()
    e = errors(long_oracle, (N,), P.conservative(EOS, a1 * 1000, (1 - a1) * 1.0, [0 * w], 15.0 + 1.5 * w, a1))
    assert e[2] <= 1.1e-12, e
