"""The packed tiles of one and two long lanes (1x32, 2x64) against the
oracle: at the edges of their scoring ranges, on ragged and empty sides, on
bands that drift through many window shifts or outgrow the window, and the
tiles they fall back to outside their range."""
import numpy as np
import pytest

from paper_2309_07270_gb300 import workloads as W

pytestmark = pytest.mark.gpu
P16 = 0x100
TILES = [(1, 32), (2, 64)]


@pytest.fixture(scope="module")
def X():
    from paper_2309_07270_gb300 import build, xdrop
    build.build()
    return xdrop


def _check(X, orc, tile, w, want_tile=None):
    with X.Aligner() as al:
        al.set_tile(tile[0], tile[1] | P16)
        got = al.align(w.packed, w.read_off, w.read_len, w.pairs,
                       X.scoring(w.match, w.mismatch, w.gap, w.x))
        assert al.tile() == (want_tile or (tile[0], tile[1] | P16))
        st = al.stats()
    want = orc.align_pairs(w.packed, w.read_off, w.read_len, w.pairs, w.match, w.mismatch, w.gap,
                           w.x, nthreads=8)
    assert np.array_equal(got.view(np.int32), want.view(np.int32)), (tile, w.name)
    return st


def _scored(w, sc):
    w.match, w.mismatch, w.gap, w.x = sc
    return w


@pytest.mark.parametrize("tile", TILES, ids=lambda t: f"{t[0]}x{t[1]}")
@pytest.mark.parametrize("sc", [(1, -1, -1, 15), (1, -1, -1, 50), (2, -3, -2, 40), (1, 0, -1, 30),
                                (1, -2, -1, 506), (32, -64, -32, 383), (7, -1, -2, 0)],
                         ids=lambda s: "_".join(map(str, s)))
def test_scorings_and_ragged_ends(X, orc, tile, sc):
    _check(X, orc, tile, _scored(W.template_pairs(n_pairs=40, len_lo=800, len_hi=2500, seed=51), sc))
    _check(X, orc, tile, _scored(W.tiny_pairs(n_pairs=150, seed=52), sc))


@pytest.mark.parametrize("tile", TILES, ids=lambda t: f"{t[0]}x{t[1]}")
def test_drifting_and_outgrown_bands(X, orc, tile):
    """One read gains a base every 8: the window shifts hundreds of slots; a
    threshold of 200 outgrows every one of these windows."""
    rng = np.random.default_rng(53)
    a, b, seeds = [], [], []
    for k in range(24):
        t = rng.integers(0, 4, int(rng.integers(300, 2500))).astype(np.uint8)
        u = np.concatenate([np.append(t[q:q + 8], rng.integers(0, 4)) for q in range(0, len(t), 8)])
        u = u.astype(np.uint8)
        a.append(t if k % 2 else u)
        b.append(u if k % 2 else t)
        seeds.append((0, 0, 8))
    w = W.from_sequences(a, b, seeds, x=14)
    st = _check(X, orc, tile, w)
    assert st["overflow_tasks"] <= 12
    st = _check(X, orc, tile, w.with_x(200))
    assert st["overflow_tasks"] > 0


@pytest.mark.parametrize("tile,sc,want", [
    ((1, 32), (1, -1, -1, 1020), (2, 16 | P16)), ((2, 64), (1, -1, -1, 508), (8, 16 | P16)), ((2, 64), (1, -3, -1, 30), (8, 16)), ((1, 32), (1, -3, -1, 30), (4, 16))])
def test_fallback_outside_the_range(X, orc, tile, sc, want):
    _check(X, orc, tile, _scored(W.template_pairs(n_pairs=8, len_lo=200, len_hi=700, seed=54), sc),
           want)
