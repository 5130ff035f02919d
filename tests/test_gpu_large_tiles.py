"""The FP64 sweeps' large tiles (1 x 123 and 2 x 64 midpoints in 1D and 2D, 2 x
59 and 4 x 32 in 3D), which grids above 608 small tiles (3D: 1216) take, with
what acts at boundaries and jumps: every scheme, every boundary kind, Dirichlet
faces uniform and per face, the limiters and the SSPRK3 combine, on partial
tiles in every direction; and both sides of the 3D line, each axis deciding.
Against the oracle with the bars of tests/test_gpu_parity.py, whose own grids
are below those lines."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import Oracle  # noqa: E402
from paper_2102_05287_gb300 import problems as P  # noqa: E402
from paper_2102_05287_gb300.wcns import Solver  # noqa: E402
from tests.test_gpu_parity import EOS, assert_parity, cfl_dt, pair  # noqa: E402

TR, PER, SYM, DIR = ("transmissive",) * 2, ("periodic",) * 2, ("symmetry", "transmissive"), ("dirichlet",) * 2
GRIDS = [(12400,), (151, 110), (62, 34, 33)]


def small_tiles(n, d):
    """Small tiles of the sweep along d: 20, 17 and 31 cells in 1D, 2D, 3D."""
    return -(-n[d] // (20, 17, 31)[len(n) - 1]) * int(np.prod(n)) // n[d]


@pytest.mark.parametrize("scheme", ["pp-wcns-is", "wcns-is", "hllc1"])
@pytest.mark.parametrize("bc", [TR, PER, SYM], ids=lambda b: b[0])
@pytest.mark.parametrize("n", GRIDS, ids=str)
def test_rhs(n, bc, scheme):
    assert min(small_tiles(n, d) for d in range(len(n))) > (1216 if len(n) == 3 else 608)
    # without limiters the jumps leave the admissible set in 3D (the oracle too)
    W = P.random_admissible(n, seed=31, jumps=scheme != "wcns-is")
    o, s = pair(n, (bc,) * len(n), scheme=scheme)
    dt = cfl_dt(o, W)
    got = s.rhs(torch.from_numpy(W).cuda(), dt).cpu().numpy()
    assert_parity(got, o.rhs(W, dt), lambda X: o.rhs(X, dt), W)
    if scheme == "pp-wcns-is":
        assert s.stats()["fp64_fallbacks"] > 0  # the jumps take the FP64 limiters
    s.close()


@pytest.mark.parametrize("per_face", [False, True])
@pytest.mark.parametrize("n", GRIDS, ids=str)
def test_rhs_with_dirichlet_faces(n, per_face):
    nd = len(n)
    W = P.random_admissible(n, seed=32)
    uniform, faces = [], {}
    for d in range(nd):
        pair_ = []
        for side in range(2):
            f = np.take(W, 0 if side == 0 else -1, axis=nd - d).reshape(nd + 4, -1).copy()
            f[2 + d] *= -1.0 if side else 1.0
            pair_.append(f[:, 0])
            faces[(d, side)] = f
        uniform.append(tuple(pair_))
    kw = dict(dirichlet_face=faces) if per_face else dict(dirichlet=tuple(uniform))
    o = Oracle(n, (0.0,) * nd, (1.0,) * nd, (DIR,) * nd, **kw, **EOS)
    s = Solver(n, (0.0,) * nd, (1.0,) * nd, (DIR,) * nd, **kw, **EOS)
    dt = cfl_dt(o, W)
    got = s.rhs(torch.from_numpy(W).cuda(), dt).cpu().numpy()
    assert_parity(got, o.rhs(W, dt), lambda X: o.rhs(X, dt), W)
    s.close()


@pytest.mark.parametrize("n", GRIDS, ids=str)
def test_step(n):
    W = P.random_admissible(n, seed=33)
    o, s = pair(n, (TR, PER, TR)[:len(n)])
    dt = cfl_dt(o, W)
    Wg = torch.from_numpy(W).cuda()
    s.rk3_step(Wg, dt)
    assert_parity(Wg.cpu().numpy(), o.rk3_step(W, dt), lambda X: o.rk3_step(X, dt), W)
    s.close()


@pytest.mark.parametrize("n", [(3, 32, 38), (3, 32, 39), (32, 3, 38), (32, 3, 39), (32, 38, 3), (32, 39, 3)], ids=str)
def test_rhs_around_the_3d_line(n):
    most = max(small_tiles(n, d) for d in range(3))
    assert most == 1216 or most == 1248
    W = P.random_admissible(n, seed=34, jumps=False)
    o, s = pair(n, (TR, PER, TR))
    dt = cfl_dt(o, W)
    got = s.rhs(torch.from_numpy(W).cuda(), dt).cpu().numpy()
    assert_parity(got, o.rhs(W, dt), lambda X: o.rhs(X, dt), W)
    s.close()
