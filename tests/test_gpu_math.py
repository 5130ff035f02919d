"""The FP64 sweeps' reciprocal, square root and square root of a quotient
(csrc/wcns_math64.cuh) against numpy's long double, over their whole exponent
ranges, odd and even exponents and the ends of the mantissa, and against
CUDA's division and square root, bit for bit, outside them: both sides of each
range's ends, zeros, negatives, subnormals, infinities and NaN.

Bounds in units in the last place of the exact value.  Each result is one
fused multiply-add of a correction below 2^-42 of it: 1/2 for that rounding
and 0.01 for the correction's own error; the root of a quotient rounds c d
before the remainder, 2^-54 of the result or up to 1/2 more."""
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

RCP, SQRT, RATIO = 0, 1, 2
N = 1 << 20


def run(kind, a, b=None):
    ta, tb = (torch.from_numpy(np.ascontiguousarray(x)).cuda() if x is not None else None for x in (a, b))
    q = torch.empty_like(ta)
    p = lambda t: C.c_void_p(t.data_ptr()) if t is not None else None  # noqa: E731
    assert wcns.load().wcns_check_math(kind, p(ta), p(tb), p(q), a.size, None) == wcns.WCNS_OK
    torch.cuda.synchronize()
    cuda = torch.reciprocal(ta) if kind == RCP else torch.sqrt(ta if kind == SQRT else ta / tb)
    return q.cpu().numpy(), cuda.cpu().numpy()


def spread(lo, hi, rng):
    """Mantissas over [1, 2), some at its ends, times 2^e, lo <= e < hi."""
    m = 1 + rng.uniform(0, 1, N)
    k = N // 8
    m[:k] = 1 + rng.integers(0, 64, k) * 2.0 ** -52
    m[k:2 * k] = 2 - rng.integers(1, 64, k) * 2.0 ** -52
    m = np.minimum(m, 2 - 2.0 ** -52)
    return np.ldexp(m, rng.integers(lo, hi, N))


def ulps(q, exact):
    ulp = np.spacing(np.abs(exact.astype(np.float64))).astype(np.longdouble)
    return float((np.abs(q.astype(np.longdouble) - exact) / ulp).max())


def test_reciprocal():
    rng = np.random.default_rng(1)
    b = spread(-1022, 1021, rng) * rng.choice([-1.0, 1.0], N)
    q, _ = run(RCP, b)
    assert ulps(q, 1 / b.astype(np.longdouble)) <= 0.51


def test_square_root():
    rng = np.random.default_rng(2)
    t = spread(-767, 769, rng)
    q, _ = run(SQRT, t)
    assert ulps(q, np.sqrt(t.astype(np.longdouble))) <= 0.51


def test_square_root_of_a_quotient():
    rng = np.random.default_rng(3)
    n, d = spread(-447, 449, rng), spread(-447, 449, rng)
    k = N // 2  # as in c^2 = n / d: comparable exponents
    n[:k] = d[:k] * np.exp(rng.uniform(-40, 40, k))
    ok = (n >= 2.0 ** -447) & (n < 2.0 ** 449)
    q, _ = run(RATIO, n[ok], d[ok])
    assert ulps(q, np.sqrt(n[ok].astype(np.longdouble) / d[ok].astype(np.longdouble))) <= 1.01


def same(x, y):
    return (x.view(np.int64) == y.view(np.int64)) | (np.isnan(x) & np.isnan(y))


def test_outside_the_ranges():
    s = [0.0, 5e-324, 1e-310, np.finfo(np.float64).max, np.inf, np.nan]
    edge = lambda *e: [np.nextafter(2.0 ** k, -np.inf) if w < 0 else 2.0 ** k for k, w in e]  # noqa: E731
    v = np.array(s + edge((-1022, -1), (1021, 1), (1022, 1)))
    q, ref = run(RCP, np.concatenate([v, -v]))
    assert same(q, ref).all()
    v = np.array(s + edge((-767, -1), (769, 1), (-1022, 1)) + [-1.0, -2.0 ** 500])
    q, ref = run(SQRT, np.concatenate([v, -v[:6]]))
    assert same(q, ref).all()
    out = np.array(s + [-x for x in s] + edge((-447, -1), (449, 1)) + [-3.0])
    inn = np.array([1.0, 7.0, 2.0 ** -447, np.nextafter(2.0 ** 449, 0)])
    for x, y in ((out, np.concatenate([out, inn])), (inn, out)):
        a, b = np.meshgrid(x, y)
        q, ref = run(RATIO, a.ravel(), b.ravel())
        assert same(q, ref).all(), [(w, z) for w, z, k in zip(a.ravel(), b.ravel(), same(q, ref)) if not k][:5]


def test_bad_arguments():
    lib, E = wcns.load(), wcns.WCNS_E_INVALID_ARG
    assert lib.wcns_check_math(3, None, None, None, 0, None) == E
    assert lib.wcns_check_math(-1, None, None, None, 0, None) == E
    assert lib.wcns_check_math(0, None, None, None, -1, None) == E
    assert lib.wcns_check_math(2, None, None, None, 4, None) == E
    assert lib.wcns_check_math(1, None, None, None, 0, None) == wcns.WCNS_OK
