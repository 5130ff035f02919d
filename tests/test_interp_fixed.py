"""The fixed-point / FP32-pair WCNS-IS interpolation of the FP64 sweeps
(csrc/wcns_isw.cuh), built for the host and compared with the printed
formula in long double.

Bound, in units of 2^-53 (scale + |u|), for every value the routine decides:
1/2 for the weights (its own acceptance test), 0.7 for the inputs' truncation
to 2^-54 of the largest (the linear weights' absolute sum is at most 1.4, and
the largest input is accepted up to scale + |u|), and as much again for the
weights' response to that truncation: 2 together.  Stencils of constants must
give exactly zero, and values it does not decide are left to FP64.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2102_05287_gb300", "csrc")
FAMILIES = ["smooth", "noisy", "random", "jump", "noise", "zeros_jump", "extremum", "ulps", "floor"]

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include "wcns_isw.cuh"
typedef long double Q;
static Q beta(Q x, Q y) { return Q(13) / 12 * x * x + y * y / 4; }
static Q is(Q a, Q b, Q c, Q d, Q e, Q eps) {
  Q s0 = (c + d) / 2, s1 = (3 * c - b) / 2, s2 = (3 * c + 6 * d - e) / 8, s3 = (3 * a - 10 * b + 15 * c) / 8;
  Q tau = beta(e - 4 * d + 6 * c - 4 * b + a, e - 2 * d + 2 * b - a), r01 = tau / (beta(b - 2 * c + d, b - d) + eps);
  Q w0 = Q(15) / 32 * (1 + tau / ((c - d) * (c - d) + eps) * r01), w1 = Q(5) / 32 * (1 + tau / ((b - c) * (b - c) + eps) * r01);
  Q w2 = Q(10) / 32 * (1 + tau / (beta(c - 2 * d + e, 3 * c - 4 * d + e) + eps));
  Q w3 = Q(2) / 32 * (1 + tau / (beta(a - 2 * b + c, a - 4 * b + 3 * c) + eps));
  return (w0 * s0 + w1 * s1 + w2 * s2 + w3 * s3) / (w0 + w1 + w2 + w3);
}
int main(int argc, char **argv) {
  const int fam = atoi(argv[1]);
  const long n = atol(argv[2]);
  std::mt19937_64 g(fam + 1);
  std::uniform_real_distribution<double> u(0, 1);
  auto lg = [&](double a, double b) { return exp(log(a) + (log(b) - log(a)) * u(g)); };
  long decided = 0, pairs = 0;
  double worst = 0;
  for (long i = 0; i < n; ++i) {
    double U[6];
    const double scale = lg(1e-8, 1e4), amp = scale * lg(1e-14, 1), kh = lg(1e-3, 1.5), p1 = 6.283 * u(g), p2 = 6.283 * u(g);
    const double eps = i % 4 ? 1e-40 : lg(1e-60, 1e-6);
    auto sm = [&](double x) { return sin(kh * x + p1) + .5 * sin(2.3 * kh * x + p2); };
    for (int j = 0; j < 6; ++j) {
      const double x = j - 2;
      double v = 0;
      if (fam == 0) v = amp * sm(x);
      if (fam == 1) v = amp * sm(x) + scale * 1e-16 * (2 * u(g) - 1);
      if (fam == 2) v = amp * (2 * u(g) - 1);
      if (fam == 3) v = amp * 1e-3 * sm(x);
      if (fam == 4) v = scale * 1e-15 * (2 * u(g) - 1);
      if (fam == 6) v = amp * ((x - .5 - 1e-3 * u(g)) * (x - .501) - .25) + amp * 1e-3 * x * x * x;
      if (fam == 7) v = scale * 2.22e-16 * (int)(u(g) * 5 - 2);
      if (fam == 8) v = amp * 1e-10 * sm(x);
      U[j] = v;
    }
    if (fam == 3 || fam == 5) {
      const int at = 1 + (int)(5 * u(g));
      for (int j = at; j < 6; ++j) U[j] += amp;
    }
    const double z = U[2];
    for (int j = 0; j < 6; ++j) U[j] -= z;
    double v[2];
    const int r = wcns::isw::interpolate(U[0], U[1], U[3], U[4], U[5], 4 * eps, (float)scale, v[0], v[1]);
    const Q x[2] = {is(U[0], U[1], 0, U[3], U[4], eps), is(U[5], U[4], U[3], 0, U[1], eps)};
    pairs += (r >> 2) & 1;
    for (int s = 0; s < 2; ++s) {
      if (!(r >> s & 1)) continue;
      ++decided;
      const double e = (double)(fabsl(v[s] - x[s]) / (1.1102230246251565e-16L * (scale + fabsl(x[s]))));
      if (!(e <= worst)) worst = e;
    }
  }
  double a = 1, b = 1;
  const int r = wcns::isw::interpolate(0, 0, -0.0, 0, 0, 4e-40, 1.0f, a, b);
  printf("%.17g %ld %ld %d\n", worst, decided, pairs, r == 3 && a == 0 && b == 0);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("isw")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")], check=True)
    return str(d / "t")


@pytest.mark.parametrize("fam", range(len(FAMILIES)), ids=FAMILIES)
def test_decided_values_within_the_bound(program, fam):
    n = 40000
    worst, decided, pairs, zeros = subprocess.run([program, str(fam), str(n)], check=True, capture_output=True, text=True).stdout.split()
    assert float(worst) <= 2.0
    assert int(zeros) == 1
    # the routine has to carry the common stencils: noise and smooth waves
    if FAMILIES[fam] in ("smooth", "noisy", "noise", "ulps", "floor"):
        assert int(decided) > 0.85 * 2 * n
    if FAMILIES[fam] in ("smooth", "random"):
        assert int(pairs) > 0.1 * n
