"""Serving requests whose scorings fit the packed tiles' 16 bits but not lanes of
32 slots: they stay off the second tier, before, after and between others."""
import numpy as np
import pytest

from paper_2309_07270_gb300 import workloads as W

pytestmark = pytest.mark.gpu
SHORT = (1, -1, -1, 50)
# just inside and just outside x + 2 match + 2|gap| <= 1023, and the 16-bit limit
SCORINGS = [(16, -16, -32, 927), (16, -16, -32, 928), (20, -24, -40, 960), (1, 0, -100, 1535)]


@pytest.mark.parametrize("tile", [None, (2, 32 | 0x100)], ids=["default", "forced"])
def test_scorings_between_16_and_32_slot_lanes(orc, tile):
    from paper_2309_07270_gb300 import build
    from paper_2309_07270_gb300 import xdrop as X
    build.build()
    w = W.template_pairs(n_pairs=120, len_lo=300, len_hi=2000, seed=91)
    ctx = X.xdrop_init(0, 0, X.XDROP_MODE_SERVE)
    try:
        if tile:
            X.xdrop_set_tile(ctx, *tile)
        X.xdrop_load_reads(ctx, w.packed, w.read_off, w.read_len)
        jobs = []
        for sc in [SHORT, SCORINGS[0], SHORT, SCORINGS[1], SHORT] + SCORINGS * 2:
            out = np.zeros(w.n_pairs, X.RESULT_DTYPE)
            jobs.append((sc, out, X.xdrop_submit_pairs(ctx, w.pairs, X.scoring(*sc), out)))
        for _, _, t in jobs:
            X.xdrop_sync(ctx, t, 60_000_000_000)
        st = X.xdrop_get_serve_stats(ctx)
    finally:
        X.xdrop_free(ctx)
    for sc, out, _ in jobs:
        want = orc.align_pairs(w.packed, w.read_off, w.read_len, w.pairs, *sc, nthreads=8)
        assert np.array_equal(out.view(np.int32), want.view(np.int32)), sc
    # bands of x / |gap| < 30 slots fit 64: only what outgrows them is handed on
    assert st["spill_reserved"] < 60 and st["wide_passes"] == 0
