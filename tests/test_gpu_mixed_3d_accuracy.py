"""The mixed 3D sweeps call their interpolations instead of inlining them, and
a returned quotient is rounded where an inlined one is fused into the next sum.
The step's error against FP64, over seeded waves in water around a bubble, is no
larger than that of the same kernels with the interpolations inlined, which
was ERROR (root mean square of the densities' and of the total energy's error
over that of the field, summed over the states)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2102_05287_gb300 import problems as P  # noqa: E402
from paper_2102_05287_gb300.wcns import Solver  # noqa: E402

EOS = P.WORKLOAD_EOS
TR = ("transmissive", "transmissive")
ERROR = (1.630e-9, 2.270e-9)


def state(n, seed):
    rng = np.random.default_rng(seed)
    X = np.meshgrid(*[(np.arange(n) + 0.5) / n] * 3, indexing="ij")

    def f():
        g = 0.0
        for _ in range(4):
            k = rng.integers(1, 5, 3) * rng.choice([-1, 1], 3)
            g = g + rng.uniform(0.3, 1.0) * np.sin(2 * np.pi * sum(a * x for a, x in zip(k, X)) + rng.uniform(0, 6.283))
        return g / 4

    r = np.sqrt(sum((x - 0.5) ** 2 for x in X))
    a1 = 1 - (1e-6 + (1 - 2e-6) * 0.5 * (1 - np.tanh((r - 0.25) * n)))
    p = np.where(r < 0.25, 1e5, 1e8 * (1 + 0.05 * f()))
    return P.conservative(EOS, a1 * 1000.0, 1 - a1, [2 * f() for _ in range(3)], p, a1)


def test_no_less_accurate_than_inlined():
    total = np.zeros(7)
    for n in (40, 64):
        for seed in range(16):
            W, out = state(n, seed), []
            for precision in ("mixed", "fp64"):
                s = Solver((n,) * 3, (0.0,) * 3, (1.0,) * 3, (TR,) * 3, precision=precision, **EOS)
                out.append(s.rk3_step(torch.from_numpy(W).cuda(), 0.3 / (3 * 4000.0 * n)).reshape(7, -1))
                s.close()
            total += ((out[0] - out[1]).norm(dim=1) / out[1].norm(dim=1)).cpu().numpy()
    assert total[0] <= ERROR[0] and total[5] <= ERROR[1], total
