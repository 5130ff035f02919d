"""Repeated steps of small grids, whose kernels are launched before their
predecessor has ended, against the batched path, which launches none early:
direct and replayed steps have to agree bit for bit, and both with the batched
problem to the 1e-14 of tests/test_gpu_batch.py, on both sides of the 304-block line (FP64 tiles of 20 cells in 1D, 17 a
line in 2D; mixed tiles of 122 and of 4 x 58)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2102_05287_gb300 import problems as P  # noqa: E402
from paper_2102_05287_gb300.wcns import Batch, Solver  # noqa: E402
from tests.test_gpu_parity import relerr  # noqa: E402

EOS = P.WORKLOAD_EOS
TR = ("transmissive", "transmissive")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [(7,), (200,), (6080,), (6081,), (40000,), (17, 5), (61, 70), (71, 73), (200, 190)])
def test_repeated_steps_equal_the_batched_path(n, precision):
    nd, steps = len(n), 12
    W = P.random_admissible(n, seed=sum(n), jumps=False)
    lo, hi = np.zeros((1, nd)), np.ones((1, nd))
    if nd == 1:
        b = Batch(n, lo[:, 0], hi[:, 0], "transmissive", "transmissive", precision=precision, **EOS)
    else:
        b = Batch.grids([n], lo, hi, (TR,) * nd, precision=precision, **EOS)
    ref = torch.from_numpy(W.reshape(nd + 4, -1).copy()).cuda()
    t = torch.zeros(1, dtype=torch.float64, device="cuda")
    s = Solver(n, (0.0,) * nd, (1.0,) * nd, (TR,) * nd, precision=precision, **EOS)
    replay, direct = torch.from_numpy(W).cuda(), torch.from_numpy(W).cuda()
    s.profile_enable(4096)  # per-kernel timing: direct launches
    td = s.advance_steps(direct, steps, cfl=0.4)
    s.profile_enable(0)
    tr = s.advance_steps(replay, steps, cfl=0.4)
    b.advance(ref, steps, cfl=0.4, t=t)
    assert s.stats()["nonfinite"] == 0
    assert torch.equal(direct, replay) and td == tr
    ref, got = ref.cpu().numpy(), replay.cpu().numpy().reshape(ref.shape)
    assert relerr(got, ref).max() <= 1e-14, relerr(got, ref)
    assert abs(float(t[0]) - tr) <= 1e-14 * tr
    s.close()
    b.close()
