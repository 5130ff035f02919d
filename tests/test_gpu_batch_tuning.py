"""The batch autotuner times each launch once: a batch whose work lists are
shorter than the number of SMs has one grid per tile length (three in 1D, one
in 2D), whatever the blocks per SM, and the first advance of a batch tries no
more.  A trial is one reduction and at most three steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2102_05287_gb300 import problems as P  # noqa: E402
from paper_2102_05287_gb300.wcns import Batch  # noqa: E402


def tuning_launches(b, W):
    b.advance(W, 1, cfl=0.5)
    first = b.launches()
    b.advance(W, 1, cfl=0.5)
    assert b.tuning() is not None and b.stats()["nonfinite"] == 0
    n = first - (b.launches() - first)  # launches of the first call beyond the second's
    b.close()
    return n


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_small_batches_try_each_launch_once(precision):
    rb = P.riemann_batch(nprob=16, seed=3, nmin=20, nmax=400)
    b = Batch(rb.sizes, np.zeros(16), np.ones(16), "transmissive", "transmissive", precision=precision, **rb.eos)
    assert tuning_launches(b, torch.from_numpy(rb.W).cuda()) <= 3 * (1 + 3 * 4)
    gb = P.bubble_batch_2d(nprob=8, seed=3, nmin=8, nmax=40)
    b = Batch.grids(gb.sizes, gb.lo, gb.hi, (("transmissive",) * 2,) * 2, precision=precision, **gb.eos)
    assert tuning_launches(b, torch.from_numpy(gb.W).cuda()) <= 1 + 3 * 7


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_large_batches_stop_where_it_gets_slower(precision):
    """Tiles for every SM many times over: fewer blocks an SM are slower, and
    after the limit and one or two more grids of a tile length none is tried."""
    rb = P.riemann_batch(nprob=1500, seed=3, nmin=500, nmax=1500)
    b = Batch(rb.sizes, np.zeros(1500), np.ones(1500), "transmissive", "transmissive", precision=precision, **rb.eos)
    assert tuning_launches(b, torch.from_numpy(rb.W).cuda()) <= 7 * (1 + 3 * 4)
