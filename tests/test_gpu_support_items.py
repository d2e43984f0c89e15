"""The support term from shared memory with more work items than two rounds of
its warps (152 SMs x 24 warps), which are then taken by count: short rows,
whole rows of up to 128 entries and the slices of longer ones, three times in a
row, since the last block sets the counts back.  Reference and tolerance as
in test_gpu_step_edges: fp32 sums against fp64, 1e-5.
"""
import numpy as np
import pytest

from paper_2608_21607_gb300 import nmd as N
from paper_2608_21607_gb300 import workloads as WL

from gpu_common import rel, require_gpu
from test_gpu_tc import pieces

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,longest", [(7000, 3), (7296, 1), (7297, 1), (15000, 40), (20001, 300)])
@pytest.mark.parametrize("r,K", [(16, 700), (32, 3200)])
def test_items_by_count(r, K, m, longest):
    require_gpu()
    g = np.random.default_rng([r, m])
    counts = 1 + np.minimum(g.integers(0, longest, m), g.integers(0, longest, m))
    starts = g.integers(0, K - counts)                 # a run of columns per row
    ptr = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    rows = np.repeat(np.arange(m), counts)
    cols = (np.repeat(starts, counts) + np.arange(ptr[-1]) - np.repeat(ptr[:-1], counts)).astype(np.int32)
    S = WL.CSR(m, K, ptr, cols, (0.5 + g.random(ptr[-1])).astype(np.float32))
    W, H = WL.init_factors(m, K, r, r)
    sol = N.Solver(S, r, block_rows=m, block_cols=K, precision=N.NMD_BF16)
    sol.set_factors(W, H)
    Mo, Qo = pieces(W)[0].astype(np.float64), pieces(np.ascontiguousarray(H.T))[0].astype(np.float64)
    c = S.vals - np.minimum(0, np.einsum("ij,ij->i", Mo[rows], Qo[cols]))
    want = np.add.reduceat(c[:, None] * Qo[cols], ptr[:-1], axis=0)
    for _ in range(3):
        got = sol.support_term(N.NMD_COL, 0, N.NMD_STOCH)
        sol.sync()
        assert rel(got.cpu().numpy()[:, :r], want) <= 1e-5
