"""Small grids take sweep tiles with one component of one midpoint a thread (in
3D a quarter of them); grids above 608 of those tiles (3D: 1216) take the
large ones.  Both sides of that line, and of the small tiles' edges (21
midpoints in 1D, 18 in 2D, 32 in 3D: 20, 17 and 31 cells a tile), against the oracle with the bars of tests/test_gpu_parity.py, under
every boundary kind and scheme the sweeps have."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2102_05287_gb300 import problems as P  # noqa: E402
from tests.test_gpu_parity import assert_parity, cfl_dt, pair  # noqa: E402

SIZES = [(1,), (20,), (21,), (41,), (12160,), (12161,), (17, 3), (18, 35), (35, 18), (101, 101), (102, 102), (31, 4, 5), (32, 3, 33),
         (3, 35, 35), (3, 34, 36)]


@pytest.mark.parametrize("scheme", ["pp-wcns-is", "hllc1"])
@pytest.mark.parametrize("bc", [("transmissive", "transmissive"), ("periodic", "periodic"), ("symmetry", "transmissive")])
@pytest.mark.parametrize("n", SIZES)
def test_rhs_around_the_tile_choice(n, bc, scheme):
    if bc[0] == "symmetry" and min(n) < 3:
        pytest.skip("symmetry needs three cells")
    o, s = pair(n, (bc,) * len(n), scheme=scheme)
    W = P.random_admissible(n, seed=len(n) + n[0], jumps=False)
    dt = cfl_dt(o, W)
    L = s.rhs(torch.from_numpy(W).cuda(), dt).cpu().numpy()
    assert_parity(L, o.rhs(W, dt), lambda x: o.rhs(x, dt), W)
    s.close()
