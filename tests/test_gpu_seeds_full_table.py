"""The row-wise product of seed discovery when a read's shared-memory table
fills while the other warps of its block are in their columns."""
import numpy as np
import pytest

from oracle import seeds as S

from test_gpu_seeds import X, as_candidates, gpu, pack, same  # noqa: F401

pytestmark = pytest.mark.gpu


def test_table_fills_while_other_warps_work(X):
    """Three reads of 6,000 positions with some 2,900 partners each: every
    warp of their blocks has columns left when one finds the table full."""
    rng = np.random.default_rng(13)
    hub = rng.integers(0, 4, 6000).astype(np.uint8)
    packed, off, lens = pack([hub] * 3 + [hub[i:i + 24].copy() for i in range(0, 5900, 2)])
    want = S.candidate_pairs(packed, off, lens, k=12, lo=1, hi=1024)
    assert (want["a"] == 0).sum() > 2900
    same(gpu(X, packed, off, lens, 12, 1, 1024, rowwise=True, expect_product=X.XDROP_SEEDS_SORT),
         want)
