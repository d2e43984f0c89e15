"""Block steps where the Gram chain, the update and the support term change
their split of the work, against the oracle (fp64) resp. the definition.

Gram chain at r_pad <= 64 (one launch: partials of 64 rows, up to 64 of them, added
by classes p mod 8, inverted by the last block): one partial, fewer than eight,
a remainder past eight, all 64, and blocks of more than 64 x 64 rows (longer
partials); ranks at and beside their padding.  Each step runs twice, so that
the second one starts from the counters that the first one left.  The ridge
keeps kappa(G) below 10 where the block has few rows.  Tolerances: each of the
three bf16 roundings (M, Q, P) is 1.1e-3 (rms), together 2e-3 of R, times at
most 5 through G^{-1}; 1e-4 for fp32-accurate operands.

Update: block rows at the edges of its 32-row tiles.

Support term from shared memory: blocks of one row up to the largest that fits
(200 KB of bf16 rows), rows of 1 to 130 entries, which leave entry slots past
an item's end empty; 1e-5 as fp32 sums against fp64.
"""
import numpy as np
import pytest

import oracle as O
from paper_2608_21607_gb300 import nmd as N
from paper_2608_21607_gb300 import workloads as WL

from gpu_common import rel, require_gpu, sync_oracle_to
from test_gpu_tc import pieces

pytestmark = pytest.mark.gpu

TOL = {N.NMD_BF16: 1e-2, N.NMD_FP32: 1e-4}


@pytest.fixture(scope="module", autouse=True)
def gpu():
    return require_gpu()


def _csr(m, n, per_row, seed):
    g = np.random.default_rng(seed)
    cols = [np.sort(g.choice(n, min(n, k), replace=False)) for k in per_row]
    ptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    return WL.CSR(m, n, ptr, np.concatenate(cols).astype(np.int32), (0.5 + g.random(ptr[-1])).astype(np.float32))


def _steps(m, K, r, precision, epilogue=N.NMD_EPI_Z):
    S = _csr(m, K, [2] * m, [m, K, r])
    g = np.random.default_rng([r, K, m])
    W, H = g.standard_normal((m, r)).astype(np.float32), g.standard_normal((r, K)).astype(np.float32)
    ridge = 0.25 * max(K, r)
    sol = N.Solver(S, r, block_rows=m, block_cols=K, precision=precision, epilogue=epilogue, eta=0.5, gamma=0.5,
                   ridge=ridge)
    sol.set_factors(W, H)
    orc = O.State(S, W.astype(np.float64), H.astype(np.float64),
                  O.Options(block_rows=m, block_cols=K, eta=0.5, gamma=0.5, ridge=ridge))
    for _ in range(2):
        sync_oracle_to(sol, orc)
        sol.block_update(N.NMD_COL, 0, N.NMD_STOCH)
        if epilogue == N.NMD_EPI_DELTA:   # X = M + (Z - L) Q (G + ridge I)^{-1}, not Z Q (G + ridge I)^{-1}
            G = orc.B.T @ orc.B
            damp = 0.5 * ridge * np.linalg.solve(G + ridge * np.eye(r), orc.A.T).T
        orc.block_update(N.NMD_COL, 0, N.NMD_STOCH)
        if epilogue == N.NMD_EPI_DELTA:
            orc.A += damp
        got = sol.get_state()[0]
        assert rel(got, orc.A) <= TOL[precision], rel(got, orc.A)


@pytest.mark.parametrize("precision", [N.NMD_BF16, N.NMD_FP32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("r", [3, 16, 17, 32, 33, 64])
@pytest.mark.parametrize("K", [1, 64, 65, 7 * 64, 8 * 64, 9 * 64 + 1, 64 * 64, 64 * 64 + 1, 9001])
def test_gram_chain(K, r, precision):
    _steps(70, K, r, precision)


@pytest.mark.parametrize("epilogue", [N.NMD_EPI_Z, N.NMD_EPI_DELTA], ids=["zform", "delta"])
@pytest.mark.parametrize("r", [16, 32, 64])
@pytest.mark.parametrize("m", [1, 31, 32, 33, 63, 64, 65, 20000])
def test_update_rows(m, r, epilogue):
    _steps(m, 640, r, N.NMD_BF16, epilogue)


@pytest.mark.parametrize("r,K", [(3, 1), (16, 40), (16, 6400), (20, 40), (32, 3200)])
def test_support_term_in_shared_memory(r, K):
    m = 140
    S = _csr(m, K, [1 + i % 130 for i in range(m)], [r, K])
    W, H = WL.init_factors(m, K, r, r)
    sol = N.Solver(S, r, block_rows=m, block_cols=K, precision=N.NMD_BF16)
    sol.set_factors(W, H)
    got = sol.support_term(N.NMD_COL, 0, N.NMD_STOCH)
    sol.sync()
    Mo, Qo = pieces(W)[0], pieces(np.ascontiguousarray(H.T))[0]
    D = np.zeros((m, K))
    for i in range(m):
        D[i, S.col_idx[S.row_ptr[i]:S.row_ptr[i + 1]]] = S.vals[S.row_ptr[i]:S.row_ptr[i + 1]]
    want = np.where(D > 0, D - np.minimum(0, Mo @ Qo.T), 0.0) @ Qo
    assert rel(got.cpu().numpy()[:, :r], want) <= 1e-5


@pytest.mark.parametrize("device", [True, False], ids=["device", "host"])
@pytest.mark.parametrize("m,n,r", [(1, 33, 1), (31, 32, 3), (33, 64, 16), (70, 1, 17), (129, 100, 64), (65, 90, 100),
                                   (300, 257, 256)])
def test_factors_in_and_out(m, n, r, device):
    """32-row tiles of the packed layout, from and to both orders, the device
    sources and destinations one float past the allocation's alignment; the
    momentum is cleared."""
    import torch
    S = _csr(m, n, [1] * m, [m, n])
    W, H = WL.init_factors(m, n, r, r)
    sol = N.Solver(S, r, block_rows=64, block_cols=64)
    sol.set_state(W + 1, H + 1, W, H, 3)
    if device:
        def at(x):
            b = torch.empty(x.size + 1, device="cuda")
            b[1:] = torch.from_numpy(np.ascontiguousarray(x).reshape(-1)).cuda()
            return b[1:].view(x.shape)
        sol.set_factors(at(W), at(H))
        Wo, Ho = at(np.zeros_like(W)), at(np.zeros_like(H))
        sol.get_factors_device(Wo, Ho)
        got = Wo.cpu().numpy(), Ho.cpu().numpy()
    else:
        sol.set_factors(W, H)
        got = sol.get_factors()
    assert np.array_equal(got[0], W) and np.array_equal(got[1], H)
    W2, H2, EW, EH, _ = sol.get_state()
    assert np.array_equal(W2, W) and np.array_equal(H2, H) and not EW.any() and not EH.any()
