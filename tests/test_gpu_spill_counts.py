"""xdrop_last_spills lists every extension that overflow_tasks counts, whatever
runs the longest ones."""
import numpy as np
import pytest

from paper_2309_07270_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,x", [(300, 200), (3000, 50), (3000, 200), (30000, 100)])
@pytest.mark.parametrize("tile", [None, (2, 32 | 0x100), (4, 16)], ids=["tuned", "2x32p", "4x16"])
def test_list_and_count_agree(n, x, tile):
    from paper_2309_07270_gb300 import build
    from paper_2309_07270_gb300 import xdrop as X
    build.build()
    w = W.uneven_pairs(n_pairs=n, seed=90, x=x)
    with X.Aligner() as al:
        if tile:
            al.set_tile(*tile)
        for _ in range(2):
            al.align(w.packed, w.read_off, w.read_len, w.pairs, X.scoring(1, -1, -1, x))
        spills, st = X.xdrop_last_spills(al.ctx), al.stats()
    assert len(spills) == st["overflow_tasks"] > (0 if x > 100 or tile else -1)
    assert len(np.unique(spills)) == len(spills) and (spills < 2 * n).all()


def test_a_ticket_without_pairs_counts_none():
    from paper_2309_07270_gb300 import build
    from paper_2309_07270_gb300 import xdrop as X
    build.build()
    w = W.uneven_pairs(n_pairs=300, seed=90, x=700)
    sc = X.scoring(1, -1, -1, 700)
    with X.Aligner() as al:
        al.align(w.packed, w.read_off, w.read_len, w.pairs, sc)
        assert al.stats()["overflow_tasks"] > 0 and al.stats()["wide_tasks"] > 0
        al.align(w.packed, w.read_off, w.read_len, w.pairs[:0], sc)
        st = al.stats()
        assert st["tasks"] == st["overflow_tasks"] == st["wide_tasks"] == 0
        assert len(X.xdrop_last_spills(al.ctx)) == 0
