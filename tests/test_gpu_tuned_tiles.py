"""A small job of a scoring that needs 32-bit cells is tuned among all tiles,
however narrow its band: its longest extensions want the one of most lanes."""
import numpy as np
import pytest

from paper_2309_07270_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_small_32bit_job_takes_the_short_diagonal(orc):
    from paper_2309_07270_gb300 import build
    from paper_2309_07270_gb300 import xdrop as X
    build.build()
    w = W.template_pairs(n_pairs=1500, len_lo=1000, len_hi=3000, seed=5)
    with X.Aligner() as al:
        got = al.align(w.packed, w.read_off, w.read_len, w.pairs, X.scoring(100, -200, -60, 900))
        assert al.tile() == (32, 4)  # 2.3 ms; the 64-slot tiles, nearest to x / |gap|, 2.6 to 3.6
    want = orc.align_pairs(w.packed, w.read_off, w.read_len, w.pairs, 100, -200, -60, 900,
                           nthreads=8)
    assert np.array_equal(got.view(np.int32), want.view(np.int32))
