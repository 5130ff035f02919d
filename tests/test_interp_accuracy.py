"""The fixed-point / FP32-pair WCNS-IS interpolation of the FP64 sweeps
(csrc/wcns_isw.cuh, built for the host) is no less accurate than the printed
formula in FP64 that it stands for: over stencils whose deviations are as
large as the field, and of smooth waves on an offset, the midpoint value
v = x_i + u has an error (against long double) of no larger root mean square
than with u from the FP64 formula, over all values, decided or left to FP64.
Where both are rounded alike the two figures are equal up to sampling: 1 %
for 200000 stencils, two values each."""
import shutil
import subprocess

import pytest

from tests.test_interp_fixed import CSRC, SOURCE

FAMILIES = ["wave", "crossing", "offset"]

MAIN = r"""
static double b4(double a, double c, double e) { return fma(13.0 / 3 * a, a, fma(c, c, e)); }
// the FP64 formula of the deviations from the upwind node
static double f64(double um2, double um1, double up1, double up2, double e) {
  const double b01 = b4(um1 + up1, um1 - up1, e), b2 = b4(up2 - 2 * up1, up2 - 4 * up1, e), b3 = b4(um2 - 2 * um1, um2 - 4 * um1, e);
  const double ta = (um2 + up2) - 4 * (um1 + up1), tc = (up2 - um2) + 2 * (um1 - up1), tau = fma(13.0 / 3 * ta, ta, tc * tc);
  const double r = tau / b01, v0 = fma(tau / fma(4 * up1, up1, e), r, 1), v1 = fma(tau / fma(4 * um1, um1, e), r, 1);
  const double v2 = 1 + tau / b2, v3 = 1 + tau / b3;
  return (5.0 / 32 * (v0 * 1.5 * up1 - v1 * .5 * um1 + v2 * fma(1.5, up1, -.25 * up2)) + 1.0 / 16 * v3 * fma(-1.25, um1, .375 * um2)) /
         (15.0 / 32 * v0 + 5.0 / 32 * v1 + 5.0 / 16 * v2 + 1.0 / 16 * v3);
}
int main(int, char **argv) {
  const int fam = atoi(argv[1]);
  std::mt19937_64 g(fam + 1);
  std::uniform_real_distribution<double> r(0, 1);
  long n = 200000, decided = 0;
  Q s[2] = {0, 0};
  for (long i = 0; i < n; ++i) {
    const double A = exp(log(1e-8) + log(1e10) * r(g)), kh = exp(log(1e-2) + log(25.) * r(g)), p = 6.283 * r(g), x0 = r(g);
    double U[6], md = 0, v[2];
    for (int j = 0; j < 6; ++j) {
      const double x = j - 2;
      U[j] = fam == 1 ? A * sin(kh * (x - x0)) : A * ((fam == 2 ? 10 * x0 : 0) + sin(kh * x + p) + .3 * sin(2.3 * kh * x));
    }
    const double z = U[2];
    for (int j = 0; j < 6; ++j) U[j] -= z, md = fmax(md, fabs(U[j]));
    const Q x[2] = {is(U[0], U[1], 0, U[3], U[4], 1e-40L), is(U[5], U[4], U[3], 0, U[1], 1e-40L)};
    const double f[2] = {f64(U[0], U[1], U[3], U[4], 4e-40), f64(U[5] - U[3], U[4] - U[3], -U[3], U[1] - U[3], 4e-40) + U[3]};
    const int ok = wcns::isw::interpolate(U[0], U[1], U[3], U[4], U[5], 4e-40, SCALE, v[0], v[1] EXTRA);
    for (int k = 0; k < 2; ++k) {
      const double u = ok >> k & 1 ? v[k] : f[k];
      decided += ok >> k & 1;
      const Q a = ((Q)(z + u) - (z + x[k])) / (fabs(z) + md), b = ((Q)(z + f[k]) - (z + x[k])) / (fabs(z) + md);
      s[0] += a * a, s[1] += b * b;
    }
  }
  printf("%.6g %.6g %.6g\n", (double)sqrtl(s[0] / (2 * n)), (double)sqrtl(s[1] / (2 * n)), decided / (2. * n));
}
"""


def build(d, scale, extra):
    if not shutil.which("g++"):
        pytest.skip("needs g++")
    (d / "t.cpp").write_text(SOURCE[:SOURCE.index("int main")] + MAIN.replace("SCALE", scale).replace("EXTRA", extra))
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")], check=True)
    return str(d / "t")


def figures(program, fam):
    return [float(x) for x in subprocess.run([program, str(fam)], check=True, capture_output=True, text=True).stdout.split()]


@pytest.mark.parametrize("fam", range(len(FAMILIES)), ids=FAMILIES)
def test_no_less_accurate_than_the_fp64_formula(tmp_path, fam):
    """Scale: the value and the largest deviation, what v can be rounded at."""
    new, fp64, decided = figures(build(tmp_path, "(float)(fabs(z) + md)", ""), fam)
    assert decided > 0.3
    assert new <= 1.01 * fp64, (new, fp64)


@pytest.mark.parametrize("fam", range(len(FAMILIES)), ids=FAMILIES)
def test_velocities_no_less_accurate_than_the_fp64_formula(tmp_path, fam):
    """As the sweeps call it for a velocity: the value, and own = UNIT."""
    new, fp64, decided = figures(build(tmp_path, "(float)fabs(z)", ", wcns::isw::UNIT"), fam)
    assert decided > 0.3
    assert new <= 1.01 * fp64, (new, fp64)
