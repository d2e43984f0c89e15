"""Kernel timing: every step counts one Gram chain, however many parts of it
are timed (at r_pad >= 128 its partial sums run ahead on another stream), one
dense launch and one support term."""
import pytest

from paper_2608_21607_gb300 import nmd as N
from paper_2608_21607_gb300 import workloads as WL

from gpu_common import PREC_NAMES, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [N.NMD_BF16, N.NMD_FP32, N.NMD_SIMT], ids=lambda p: PREC_NAMES[p])
@pytest.mark.parametrize("r", [3, 64, 100, 200])
def test_one_launch_per_step_and_class(r, prec):
    require_gpu()
    S = WL.connectome(4000, seed=2)
    W, H = WL.init_factors(4000, 4000, r, 2)
    sol = N.Solver(S, r, block_rows=2048, block_cols=2048, precision=prec, eta=0.3, gamma=0.5)
    sol.set_factors(W, H)
    sol.profile(True)
    sol.sweep()   # two column and two row blocks
    for cls in (N.NMD_K_GRAM, N.NMD_K_DENSE, N.NMD_K_SPARSE):
        ms, launches = sol.profile_read(cls)
        assert launches == 4 and ms > 0, (cls, ms, launches)
