"""The losses of factors whose squares leave the range of fp32 sums.

L is one power of two, c on the even columns and -c on the odd ones, so that it
is exact in every mode; the support lies on odd columns.  Sums over any number
of columns are right in fp64 while a 128-column chunk's fp32 sum is finite
(c = 2^58 and 2^60; a row's sum of c^2 is past 3.4e38 in both); beyond it (2^66)
the losses are infinite.  A factor entry that is not a number shows in the
objective.  Tolerance: 1e-6, fp32 sums of at most 128 equal terms.
"""
import math

import numpy as np
import pytest

from paper_2608_21607_gb300 import nmd as N
from paper_2608_21607_gb300 import workloads as WL

from gpu_common import PREC_NAMES, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    return require_gpu()


def _case(m, n, r, e):
    cols = (2 * (np.arange(m) * 37 % (n // 2)) + 1).astype(np.int32)
    S = WL.CSR(m, n, np.arange(m + 1, dtype=np.int64), cols, np.full(m, 3.0, np.float32))
    W, H = np.zeros((m, r), np.float32), np.zeros((r, n), np.float32)
    W[:, r // 2] = 2.0 ** (e // 2)
    H[r // 2] = np.where(np.arange(n) % 2 == 0, 1.0, -1.0) * 2.0 ** (e - e // 2)
    return S, W, H


@pytest.mark.parametrize("prec", [N.NMD_BF16, N.NMD_FP32, N.NMD_SIMT], ids=lambda p: PREC_NAMES[p])
@pytest.mark.parametrize("m,n,r,e", [(200, 139255, 3, 58), (300, 5001, 64, 60), (130, 5001, 128, 60),
                                     (300, 5001, 256, 60), (300, 5001, 3, 66), (300, 5001, 64, 66)])
def test_large_entries(m, n, r, e, prec):
    S, W, H = _case(m, n, r, e)
    sol = N.Solver(S, r, block_rows=512, block_cols=512, precision=prec)
    sol.set_factors(W, H)
    got = sol.loss()
    c2, pos, fro = 4.0 ** e, m * ((n + 1) // 2), 3.0 * math.sqrt(m)
    assert got["wjd"] == pytest.approx(1.0, rel=1e-6)
    assert got["sum_relu"] == pytest.approx(pos * 2.0 ** e, rel=1e-6)
    if e < 64:
        assert got["sum_relu2"] == pytest.approx(pos * c2, rel=1e-6)
        assert got["obj"] == pytest.approx(math.sqrt(pos * c2 + m * (3.0 + 2.0 ** e) ** 2) / fro, rel=1e-6)
        assert got["rmse"] == pytest.approx(math.sqrt(pos * c2 + 9.0 * m) / fro, rel=1e-6)
    else:
        assert got["sum_relu2"] == math.inf and got["obj"] == math.inf and got["rmse"] == math.inf


@pytest.mark.parametrize("prec", [N.NMD_BF16, N.NMD_FP32, N.NMD_SIMT], ids=lambda p: PREC_NAMES[p])
@pytest.mark.parametrize("r", [3, 64])
def test_nan_is_not_a_perfect_fit(r, prec):
    S, W, H = _case(200, 600, r, 4)
    W[70, r // 2] = math.nan
    sol = N.Solver(S, r, block_rows=128, block_cols=128, precision=prec)
    sol.set_factors(W, H)
    assert math.isnan(sol.loss()["obj"])
