"""max(|u_d| + c): the reduction's FP32 screening must not pass over the cell
that holds the maximum, for every gas that wcns_create accepts.  One faster cell
at the end of a grid of equal ones, whose maximum every thread knows by then:
- a gas with gamma_g near 1, whose Gamma = dr alpha1 + r2 is a small difference
  of large numbers near alpha1 = 1, near rho c^2 = 0, where pbar's error in
  FP32 can exceed E - pbar (without an allowance the speed comes out up to 25 %
  low for gamma_g = 1.0003);
- densities and energies at the ends of FP32's range, and partial densities
  whose sum cancels.
The faster cell is 1 % ahead.  A grid of that one cell is not screened, so the
two results have to be equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2102_05287_gb300.wcns import Solver  # noqa: E402

N = 400000  # more cells than the reduction has threads (1216 blocks of 256)
GL, PINF = 4.4, 6e8


def fastest(gamma_g, a1, rho1, rho2, m, c_fast):
    """The reduction's maximum over N cells of sound speed 0.99 c_fast and
    momentum m with one of c_fast among them, and that cell's own."""
    r1, r2 = 1 / (GL - 1), 1 / (gamma_g - 1)
    G = np.longdouble(a1) * r1 + (1 - np.longdouble(a1)) * r2
    rho = np.longdouble(rho1) + rho2
    pbar = np.longdouble(a1) * (GL * PINF * r1) / (G + 1)

    def energy(c):  # c^2 = (1 + 1/Gamma) (rho e - pbar) / (Gamma rho)
        return float(0.5 * np.longdouble(m) ** 2 / rho + pbar + rho * np.longdouble(c) ** 2 * G * G / (G + 1))

    W = np.empty((5, N))
    W[:] = np.array([rho1, rho2, m, energy(0.99 * c_fast), a1])[:, None]
    W[3, -2] = energy(c_fast)
    out = []
    for X in (W, np.ascontiguousarray(W[:, -2:-1])):
        s = Solver((X.shape[1],), (0.0,), (1.0,), (("transmissive",) * 2,), gamma_g=gamma_g, gamma_l=GL, pinf_l=PINF)
        out.append(s.max_wavespeed(torch.from_numpy(X).cuda())[0])
        s.close()
    assert np.isfinite(out[1]) and out[1] > 0.99 * c_fast
    return out


@pytest.mark.parametrize("gamma_g", [1.00001, 1.0001, 1.0003, 1.003, 1.4])
def test_gamma_near_one(gamma_g):
    for a1 in 1 - np.geomspace(1e-6, 1e-4, 48):
        for c in (20.0, 34.0, 60.0):
            got, want = fastest(gamma_g, float(a1), 1000.0, 1e-5, 0.0, c)
            assert got == want, (a1, c, got, want)


@pytest.mark.parametrize("rho1, rho2, m, c", [(0.0, 1e38, 0.0, 1.0), (0.0, 2e38, 1e38, 0.5), (0.0, 1e31, 1e30, 3e3),
                                             (0.0, 1e-25, 1e-30, 1e3), (0.0, 1e-30, 1e-38, 1e-9),
                                             (0.0, 1e-12, 1e-20, 1e7), (1.0, -0.9999999, 0.0, 10.0)])
def test_densities_at_the_ends_of_fp32(rho1, rho2, m, c):
    # alpha1 = 0: pbar = 0, so that c is free
    got, want = fastest(1.4, 0.0, rho1, rho2, m, c)
    assert got == want, (got, want)
