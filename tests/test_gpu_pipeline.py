"""The dense kernel's pipeline where it wraps, and the losses of a graph with a
hub.

Dense kernel: steps with several 128-row tiles per CTA (60,100 rows: four) and
one to a few Q chunks per tile, so that the stages, the L and R accumulators
and the W buffers are reused within and across tiles, with ragged last tiles
and chunks; every 128-row tile of R is checked by itself.  The reference forms
P from L in fp64, the kernel from fp32 sums: a P within fp32 rounding of a
bf16 (fp32-accurate mode: second piece) boundary may round the other way,
about 1e-4 of the entries by 2^-8 (2^-16), which is below 1e-3 of a tile's R.

Losses: one row and one column of S with an entry in every place, among rows
of a few entries (the rows are walked 32 entries at a time from a list of
equal ranges, the dense pass finds them by warps); tolerances as for the
losses elsewhere: 5e-3 with bf16 operands, 1e-4 in the fp32-accurate mode.
"""
import numpy as np
import pytest

import oracle as O
from paper_2608_21607_gb300 import nmd as N
from paper_2608_21607_gb300 import workloads as WL

from gpu_common import TOL, require_gpu
from test_gpu_tc import bf16_round, pieces

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    return require_gpu()


@pytest.mark.parametrize("epi", [N.NMD_EPI_Z, N.NMD_EPI_DELTA], ids=["zform", "delta"])
@pytest.mark.parametrize("precision", [N.NMD_BF16, N.NMD_FP32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("r,K", [(16, 100), (16, 257), (32, 128), (64, 129), (64, 300), (64, 640), (128, 200),
                                 (128, 520), (256, 300)])
def test_tiles_and_chunks(r, K, precision, epi):
    m = 60100
    g = np.random.default_rng([r, K])
    S = WL.CSR(m, K, np.arange(m + 1, dtype=np.int64), g.integers(0, K, m).astype(np.int32), np.ones(m, np.float32))
    W, H = WL.init_factors(m, K, r, r)
    sol = N.Solver(S, r, block_rows=m, block_cols=K, precision=precision, epilogue=epi)
    sol.set_factors(W, H)
    got, _ = sol.block_terms(N.NMD_COL, 0, N.NMD_STOCH)
    Q = np.ascontiguousarray(H.T)
    qh, ql, ql2 = pieces(Q)
    wh, wl, _ = pieces(W)
    if precision == N.NMD_BF16:
        L = wh @ qh.T
        P = np.minimum(0, L) if epi == N.NMD_EPI_Z else -np.maximum(0, L)
        R = bf16_round(P.astype(np.float32)) @ qh
        lij = np.einsum("ij,ij->i", wh, qh[S.col_idx])
        R += (1.0 - np.minimum(0, lij))[:, None] * qh[S.col_idx]
        Qd = Q.astype(np.float64)
        R = R @ np.linalg.solve(qh.T @ qh, Qd.T @ Qd)
    else:
        L = wh @ qh.T + wh @ ql.T + wl @ qh.T
        P = np.minimum(0, L) if epi == N.NMD_EPI_Z else -np.maximum(0, L)
        ph = bf16_round(P.astype(np.float32))
        pl = bf16_round((P - ph).astype(np.float32))
        R = ph @ (qh + ql + ql2) + pl @ qh
        Qd = Q.astype(np.float64)
        lij = np.einsum("ij,ij->i", W.astype(np.float64), Qd[S.col_idx])
        R += (1.0 - np.minimum(0, lij))[:, None] * Qd[S.col_idx]
    for t in range(0, m, 128):
        e = np.linalg.norm(got[t:t + 128] - R[t:t + 128]) / np.linalg.norm(R[t:t + 128])
        assert e <= 1e-3, (t // 128, e)


@pytest.mark.parametrize("precision", [N.NMD_BF16, N.NMD_FP32, N.NMD_SIMT], ids=["bf16", "fp32", "simt"])
@pytest.mark.parametrize("r,m,n", [(3, 500, 700), (16, 1500, 1300), (64, 1500, 1300), (100, 600, 900), (256, 700, 500)])
def test_loss_with_hubs(r, m, n, precision):
    g = np.random.default_rng([r, m])
    D = np.where(g.random((m, n)) < 0.01, np.ceil(np.exp(1 + g.standard_normal((m, n)))), 0.0)
    D[m // 3] = 1.0 + g.random(n)
    D[:, n // 2] = 1.0 + g.random(m)
    D[m // 2 + 1] = 0.0     # rows without entries on both sides of the middle
    D[-1] = 0.0
    S = WL.csr_from_dense(D)
    W, H = WL.init_factors(m, n, r, r, sigma=0.5)
    sol = N.Solver(S, r, block_rows=256, block_cols=256, precision=precision)
    sol.set_factors(W, H)
    got = sol.loss()
    want = O.loss(O.Sparse.from_csr(S), W, H.T)
    for k in ("obj", "rmse", "wjd"):
        assert abs(got[k] - want[k]) <= TOL[precision] * abs(want[k]), (k, got[k], want[k])
