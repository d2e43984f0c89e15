"""The dense kernel's L buffers where every chunk changes tile: 60,100 rows are
three or four 128-row tiles per CTA, one Q chunk each, so that a buffer is
overwritten by the first product of another tile than the one whose second
product read it.  Reference and tolerance as in test_gpu_pipeline.
"""
import pytest

import test_gpu_pipeline as P
from paper_2608_21607_gb300 import nmd as N

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    return require_gpu()


@pytest.mark.parametrize("epi", [N.NMD_EPI_Z, N.NMD_EPI_DELTA], ids=["zform", "delta"])
@pytest.mark.parametrize("precision", [N.NMD_BF16, N.NMD_FP32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("r,K", [(64, 128), (80, 128)])
def test_one_chunk_per_tile(r, K, precision, epi):
    P.test_tiles_and_chunks(r, K, precision, epi)
