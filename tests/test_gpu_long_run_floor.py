"""The round-off floor of a long FP64 run: smooth interface advection on 1024
cells, 25600 SSPRK3 steps, where the scheme's own error is below 1e-14.  What
is left is the steps' rounding: 1/3 and 2/3 are both rounded down, by 2^-54
together, so that the mean of alpha1 = 1/2 loses up to 2.8e-17 a step, 7.1e-13
in all.  With W^n's product fused into the sum the other product's rounding
takes off a third of that: a mean error of 5.8e-13 over the cells."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2102_05287_gb300 import problems as P  # noqa: E402
from paper_2102_05287_gb300.wcns import Solver  # noqa: E402


def test_advection_floor():
    pr = P.advection_1d_smooth(1024)
    s = Solver(pr.n, pr.lo, pr.hi, pr.bcs, **pr.eos)
    W = torch.from_numpy(pr.W).cuda()
    t = s.advance_steps(W, int(round(pr.t_end / pr.dt_fixed)), dt_fixed=pr.dt_fixed)
    s.close()
    err = np.abs(W[-1].cpu().numpy() - pr.extra["exact"](t)).mean()
    assert err <= 6.0e-13, err
