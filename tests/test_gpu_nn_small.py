"""The nearest-neighbour search on small sets of small integers: products are
exact, ties and zeros of either sign are everywhere, and nearly every group of
32 columns improves on a row's best so far.  The first index of the largest
product is expected, as integers give it; sizes around a group, a tile and
several chunks.  A row that is not a number is nobody's neighbour.
"""
import numpy as np
import pytest

from paper_2608_21607_gb300 import nmd as N

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return require_gpu()


def _want(x):
    p = x.astype(np.int64) @ x.astype(np.int64).T
    np.fill_diagonal(p, np.iinfo(np.int64).min)
    return p.argmax(1), p.max(1)


@pytest.mark.parametrize("d", [1, 3, 17, 64, 256])
@pytest.mark.parametrize("n", [2, 31, 33, 128, 129, 700, 3001])
def test_integer_sets(torch, n, d):
    g = np.random.default_rng([n, d])
    x = g.integers(-1, 2, (n, d)).astype(np.float32)
    x[g.random(n) < 0.2] *= -0.0 if n % 2 else 0.0   # zero rows
    nn, best, _ = N.nearest_neighbors(torch.from_numpy(x).cuda())
    wn, wb = _want(x)
    assert np.array_equal(nn.cpu().numpy(), wn) and np.array_equal(best.cpu().numpy(), wb)


@pytest.mark.parametrize("n,d", [(40, 5), (700, 64)])
def test_ascending_and_nan(torch, n, d):
    x = np.zeros((n, d), np.float32)
    x[:, 0] = np.arange(1, n + 1)          # every column beats the ones before it
    nn, best, _ = N.nearest_neighbors(torch.from_numpy(x).cuda())
    assert np.array_equal(nn.cpu().numpy(), [n - 1] * (n - 1) + [n - 2])
    x[n - 1, d // 2] = np.nan
    nn, best, _ = N.nearest_neighbors(torch.from_numpy(x).cuda())
    assert np.array_equal(nn.cpu().numpy()[:n - 1], [n - 2] * (n - 2) + [n - 3])
    # (past 256 the dropped product of the second bf16 pieces counts: 2^-18)
    assert np.allclose(best.cpu().numpy()[:n - 2], np.arange(1, n - 1) * float(n - 1), rtol=2.0 ** -16, atol=0)
