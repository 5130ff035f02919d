"""The FP64 sweeps' WCNS-IS evaluation in integers and FP32 (csrc/wcns_isw.cuh)
as the device computes it, with its approximate reciprocals and reciprocal
square roots, against the printed formula in numpy's long double: every
accepted value within the bound that include/wcns.h states,
  2^-54 (s + w B + |u|) + 2.8 * 2^-54 B + 2^-53 |u|,
over the stencil families of tests/test_interp_fixed.py, for densities (s the
field's level) and for velocities (s the node's value, w = 1)."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
if np.finfo(np.longdouble).nmant < 62:
    pytest.skip("needs a long double wider than double", allow_module_level=True)

from paper_2102_05287_gb300 import wcns  # noqa: E402

Q = np.longdouble
N = 100000


def exact(a, b, c, d, e, eps):
    beta = lambda x, y: Q(13) / 12 * x * x + y * y / 4  # noqa: E731
    s = [(c + d) / 2, (3 * c - b) / 2, (3 * c + 6 * d - e) / 8, (3 * a - 10 * b + 15 * c) / 8]
    tau = beta(e - 4 * d + 6 * c - 4 * b + a, e - 2 * d + 2 * b - a)
    r = tau / (beta(b - 2 * c + d, b - d) + eps)
    w = [Q(15) / 32 * (1 + tau / ((c - d) ** 2 + eps) * r), Q(5) / 32 * (1 + tau / ((b - c) ** 2 + eps) * r),
         Q(10) / 32 * (1 + tau / (beta(c - 2 * d + e, 3 * c - 4 * d + e) + eps)),
         Q(2) / 32 * (1 + tau / (beta(a - 2 * b + c, a - 4 * b + 3 * c) + eps))]
    return sum(x * y for x, y in zip(w, s)) / sum(w)


def stencils(kind, rng):
    lg = lambda a, b: np.exp(rng.uniform(np.log(a), np.log(b), N))  # noqa: E731
    scale, x = lg(1e-8, 1e4), np.arange(-2.0, 4.0)[:, None]
    amp, kh, p = scale * lg(1e-14, 1), lg(1e-3, 1.5), rng.uniform(0, 6.283, (2, N))
    u = lambda lo=0.0, hi=1.0: rng.uniform(lo, hi, (6, N))  # noqa: E731
    sm = np.sin(kh * x + p[0]) + 0.5 * np.sin(2.3 * kh * x + p[1])
    at = rng.integers(1, 6, N)
    U = {"smooth": amp * sm, "noisy": amp * sm + scale * 1e-16 * u(-1, 1), "random": amp * u(-1, 1),
         "jump": amp * 1e-3 * sm + amp * (np.arange(6)[:, None] >= at), "noise": scale * 1e-15 * u(-1, 1),
         "zeros_jump": amp * (np.arange(6)[:, None] >= at), "extremum": amp * ((x - 0.5) * (x - 0.501) - 0.25 + 1e-3 * x ** 3),
         "ulps": scale * 2.22e-16 * np.floor(u(-2, 3)), "floor": amp * 1e-10 * sm, "crossing": scale * np.sin(kh * (x - u()[0]))}[kind]
    return U, scale


@pytest.mark.parametrize("velocity", [False, True])
@pytest.mark.parametrize("kind", ["smooth", "noisy", "random", "jump", "noise", "zeros_jump", "extremum", "ulps", "floor", "crossing"])
def test_accepted_values_within_the_stated_bound(kind, velocity):
    rng = np.random.default_rng(11)
    U, scale = stencils(kind, rng)
    eps = np.where(rng.uniform(size=N) < 0.75, 1e-40, np.exp(rng.uniform(np.log(1e-60), np.log(1e-6), N)))
    z = U[2].copy()
    D = U - z
    s = (np.abs(z) if velocity else scale).astype(np.float32).astype(np.float64)
    rows = np.stack([D[0], D[1], D[3], D[4], D[5], 4 * eps, s, np.full(N, 4194304.0 * velocity)], axis=1)
    t = torch.from_numpy(np.ascontiguousarray(rows)).cuda()
    out, bits = torch.empty(N, 2, dtype=torch.float64, device="cuda"), torch.empty(N, dtype=torch.int32, device="cuda")
    p = lambda x: C.c_void_p(x.data_ptr())  # noqa: E731
    assert wcns.load().wcns_check_interp(p(t), p(out), p(bits), N, None) == wcns.WCNS_OK
    torch.cuda.synchronize()
    out, bits = out.cpu().numpy(), bits.cpu().numpy()
    D = D.astype(Q)
    B = np.ldexp(1.0, np.frexp(np.abs(rows[:, :5]).max(axis=1))[1])
    for k, ref in enumerate((exact(*D[:5], Q(1) * eps), exact(*D[:0:-1], Q(1) * eps))):
        ok = (bits >> k & 1).astype(bool)
        m = np.abs(ref)
        bound = 2.0 ** -54 * (s + velocity * B + m + 2.8 * B) + 2.0 ** -53 * m
        err = np.abs(out[:, k] - ref)
        bad = ok & ~(err <= bound)
        assert not bad.any(), (bad.sum(), float((err / bound)[ok].max()))
    if kind in ("smooth", "floor"):
        assert (bits & 3).astype(bool).mean() > 0.3


def test_bad_arguments():
    lib, E = wcns.load(), wcns.WCNS_E_INVALID_ARG
    assert lib.wcns_check_interp(None, None, None, -1, None) == E
    assert lib.wcns_check_interp(None, None, None, 4, None) == E
    assert lib.wcns_check_interp(None, None, None, 0, None) == wcns.WCNS_OK
