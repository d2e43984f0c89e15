"""Sweeps whose deferred update walks many tiles, against the same block steps
run one after another, and errors that are raised while such an update runs.

In a sweep the rows that the next step does not read are updated beside it: at
33 <= r <= 64 (bf16) by one block per SM that draws batches of four 32-row
tiles from a counter, over the rows before and behind the next step's block.
40,000 rows are 1,122 deferred tiles, two batches for most blocks; every block
of the sweep is the next step's once, the first (no rows before it), the last
(ragged) and the middle ones.  The arithmetic of a row does not depend on the
launch that updates it, so the results are the serial steps' bit for bit.
(The last cases have blocks of at most 1,024 rows and at most one tile per SM,
where the Gram chain and the dense kernel change streams within sweeps.)

Errors: one row's momentum makes its first update overflow, so that a block of
the deferred launch reports it while others start; the sweep returns the error,
and the handle, whose counters are then used again, gives bit for bit what a
new one gives.
"""
import numpy as np
import pytest

import oracle as O
from paper_2608_21607_gb300 import nmd as N
from paper_2608_21607_gb300 import workloads as WL

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    return require_gpu()


def _two_per_row(n, seed):
    """n x n, one entry in either half of the columns of every row."""
    g = np.random.default_rng(seed)
    h = n // 2
    cols = np.stack([g.integers(0, h, n), g.integers(h, n, n)], 1).reshape(-1)
    return WL.CSR(n, n, 2 * np.arange(n + 1, dtype=np.int64), cols.astype(np.int32),
                  (0.5 + g.random(2 * n)).astype(np.float32))


def _solver(S, r, block, precision=N.NMD_BF16, **kw):
    return N.Solver(S, r, block_rows=block, block_cols=block, precision=precision, eta=0.3, gamma=0.5, **kw)


def _same(a, b):
    for x, y in zip(a.get_state()[:4], b.get_state()[:4]):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("r,n,block", [(64, 40000, 4096), (33, 40000, 4096), (50, 20001, 640), (64, 4000, 4000),
                                       (16, 40000, 4096), (128, 20001, 4096), (3, 6000, 512), (64, 6000, 1000),
                                       (64, 19456, 1024)])
def test_sweeps_equal_serial_steps(r, n, block, precision=N.NMD_BF16, **kw):
    S = _two_per_row(n, [r, n])
    W, H = WL.init_factors(n, n, r, r)
    a, b = _solver(S, r, block, precision, **kw), _solver(S, r, block, precision, **kw)
    a.set_factors(W, H)
    b.set_factors(W, H)
    orc = O.State(S, W.astype(np.float64), H.astype(np.float64), O.Options(block_rows=block, block_cols=block))
    for sweep in range(2):
        a.sweep()
        for side, k, kind in orc.sweep_steps(sweep):
            b.block_update(side, k, kind)
        a.sync()
        b.sync()
        _same(a, b)


@pytest.mark.parametrize("r,n,block", [(64, 20001, 4096), (100, 4000, 2048), (100, 20001, 4096), (256, 20001, 8192)])
def test_fp32_sweeps_equal_serial_steps(r, n, block):
    """At r_pad >= 128 the Gram partials run ahead of the dense kernel up to one
    tile per SM, beside it with more."""
    test_sweeps_equal_serial_steps(r, n, block, N.NMD_FP32)


@pytest.mark.parametrize("precision", [N.NMD_BF16, N.NMD_FP32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("r,n,block", [(64, 6000, 2048), (100, 6000, 2048), (200, 20001, 4096)])
def test_range_sweeps_equal_serial_steps(r, n, block, precision):
    """With the range search the Gram chain runs beside its pass."""
    test_sweeps_equal_serial_steps(r, n, block, precision, epilogue=N.NMD_EPI_DELTA,
                                   skip_zero_chunks=N.NMD_SKIP_RANGE)


@pytest.mark.parametrize("r,n,block", [(64, 40000, 4096), (16, 40000, 4096), (128, 20001, 4096), (256, 20001, 4096)])
@pytest.mark.parametrize("where", [0.0, 0.4, 1.0])
def test_error_during_a_deferred_update(r, n, block, where):
    S = _two_per_row(n, [r, n])
    W, H = WL.init_factors(n, n, r, r)
    zW, zH = np.zeros_like(W), np.zeros_like(H)
    a = _solver(S, r, block)
    EW = zW.copy()
    EW[int(where * (n - 1))] = 3e38
    bad = W.copy()
    bad[int(where * (n - 1))] = 3e38
    a.set_state(bad, H, EW, zH, 0)
    a.sweep()
    with pytest.raises(N.NmdError) as e:
        a.sync()
    assert e.value.status in (N.NMD_ERR_DIVERGED, N.NMD_ERR_NOT_SPD)
    b = _solver(S, r, block)
    for s in (a, b):
        s.set_state(W, H, zW, zH, 0)
        s.sweep()
        s.sync()
    _same(a, b)
