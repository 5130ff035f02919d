"""max(|u_d| + c): the reduction's FP32 screening against numpy's float64 over
every cell, on grids of several cells a thread, with the maximum anywhere, in
uniform states, and with a cell that is not admissible or not a number."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2102_05287_gb300 import problems as P  # noqa: E402
from paper_2102_05287_gb300.wcns import Solver  # noqa: E402

EOS = P.WORKLOAD_EOS


def speeds(W, nd):
    rho = W[0] + W[1]
    v = W[2:2 + nd] / rho
    r1, r2 = 1 / (EOS["gamma_l"] - 1), 1 / (EOS["gamma_g"] - 1)
    G = W[3 + nd] * (r1 - r2) + r2
    Pi = W[3 + nd] * EOS["gamma_l"] * EOS["pinf_l"] * r1
    p = (W[2 + nd] - 0.5 * (W[2:2 + nd] * v).sum(0) - Pi) / G
    return np.abs(v) + np.sqrt(((G + 1) * p + Pi) / (G * rho))


@pytest.mark.parametrize("n", [(1500, 1000), (701, 503), (1 << 21,), (120, 130, 110), (5, 3)])
@pytest.mark.parametrize("kind", ["uniform", "near", "wild", "nan", "negative"])
def test_reduction(n, kind):
    nd = len(n)
    rng = np.random.default_rng(nd)
    shape = tuple(reversed(n))
    amp = {"uniform": 0.0, "near": 1e-6}.get(kind, 0.5)
    f = lambda: 1 + amp * rng.uniform(-1, 1, shape)  # noqa: E731
    a1 = np.where(rng.uniform(size=shape) < 0.5, 1 - 1e-6, 1e-6) if kind == "wild" else np.full(shape, 1 - 1e-6)
    W = P.conservative(EOS, a1 * 1000 * f(), (1 - a1) * 10 * f(), [300 * f() for _ in n], 1e6 * f(), a1)
    flat = W.reshape(W.shape[0], -1)
    at = flat.shape[1] - 2
    if kind == "nan":
        flat[0, at] = np.nan
    if kind == "negative":
        flat[2 + nd, at] = -1e9  # rho c^2 < 0: the wave speed is not a number
    s = Solver(n, (0.0,) * nd, (1.0,) * nd, (("transmissive",) * 2,) * nd, **EOS)
    got = s.max_wavespeed(torch.from_numpy(W).cuda())[:nd]
    s.close()
    if kind in ("nan", "negative"):
        assert np.isnan(got).all()
    else:  # both within a few roundings of c: 1e-14
        np.testing.assert_allclose(got, speeds(W, nd).reshape(nd, -1).max(axis=1), rtol=1e-14)
