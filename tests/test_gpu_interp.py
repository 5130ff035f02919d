"""The FP64 sweeps' interpolation against the oracle over wave amplitudes:
constant states (nothing to interpolate), rounding-level and weak waves (FP32
weights), moderate ones (FP32 pairs), strong waves and a material jump (FP64,
the packed task list), at lengths around the tile edges.  The bars are those
of tests/test_gpu_parity.py: one SSPRK3 step within 1e-12 of the oracle, or 4
times the oracle's own 1-ulp spread.  With the jump the limiters are off (the
scheme's WCNS-IS form): at a sharp jump the flux limiter can put a cell
exactly at its tolerance, where Algorithm 4 decides on one rounding, and what
is compared here is the interpolation."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2102_05287_gb300 import problems as P  # noqa: E402
from tests.test_gpu_parity import EOS, assert_parity, cfl_dt, pair  # noqa: E402


def state(n, amp, jump):
    grid = np.meshgrid(*[(np.arange(m) + 0.5) / m for m in reversed(n)], indexing="ij")
    ph = sum((k + 1) * 2 * np.pi * x for k, x in enumerate(grid))
    w = 1 + amp * np.sin(ph)
    a1 = np.where(grid[-1] > 0.6, 1e-6, 0.7) * np.ones_like(ph) if jump else 0.7 * (2 - w) + 0 * ph
    return P.conservative(EOS, a1 * 1000 * w, (1 - a1) * 2 * w, [100 * w for _ in n], 1e6 * w, a1)


@pytest.mark.parametrize("jump", [False, True])
@pytest.mark.parametrize("amp", [0.0, 1e-15, 1e-11, 1e-7, 1e-4, 1e-2, 0.3])
@pytest.mark.parametrize("n", [(7,), (122,), (131,), (70, 5), (3, 65), (9, 7, 33)])
def test_amplitudes(n, amp, jump):
    o, s = pair(n, tuple(("periodic", "periodic") for _ in n), scheme="wcns-is" if jump else "pp-wcns-is")
    W = state(n, amp, jump)
    dt = cfl_dt(o, W)
    Wg = torch.from_numpy(W).cuda()
    s.rk3_step(Wg, dt)
    assert_parity(Wg.cpu().numpy(), o.rk3_step(W, dt), lambda x: o.rk3_step(x, dt), W)
    s.close()
