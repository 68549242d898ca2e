"""Batches whose longest extensions go to single warps beside the group
tier, with plentiful short overflow (the second group tier, or single warps
when it is little) and long overflow, against the oracle."""
import numpy as np
import pytest

from paper_2309_07270_gb300 import workloads as W

pytestmark = pytest.mark.gpu
P16 = 0x100


@pytest.fixture(scope="module")
def X():
    from paper_2309_07270_gb300 import build, xdrop
    build.build()
    return xdrop


@pytest.mark.parametrize("n,x", [(700, 50), (6000, 50), (6000, 20), (30000, 50), (3000, 110)])
def test_uneven_batches(X, orc, n, x):
    w = W.uneven_pairs(n_pairs=n, seed=70 + n % 97, x=x)
    want = orc.align_pairs(w.packed, w.read_off, w.read_len, w.pairs, 1, -1, -1, x,
                           nthreads=8).view(np.int32)
    sc = X.scoring(1, -1, -1, x)
    for tile in (None, (2, 32), (1, 32), (4, 32), (8, 8)):
        with X.Aligner() as al:
            if tile:
                al.set_tile(tile[0], tile[1] | P16)
            for _ in range(2):  # tuned, then from the graph alone
                got = al.align(w.packed, w.read_off, w.read_len, w.pairs, sc).view(np.int32)
                assert np.array_equal(got, want), (n, x, tile)
            st = al.stats()
            spills = X.xdrop_last_spills(al.ctx)
        if tile == (1, 32) and x >= 50:
            assert st["overflow_tasks"] == len(spills) > n // 20  # past the few that take a warp each
            assert len(np.unique(spills)) == len(spills) and spills.max() < 2 * n
