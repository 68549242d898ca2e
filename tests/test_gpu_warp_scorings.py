"""Single warps on the 16-bit scorings beyond their own window (the group loop on
32 lanes of 4 slots) against the oracle: both of its limits, ragged and empty
sides, drifting and outgrown bands; small batches, the allocation-free call,
and the longest extensions of a larger batch."""
import numpy as np
import pytest

from paper_2309_07270_gb300 import workloads as W

from test_gpu_warp_kernel import X, _oracle, _sc, _small, _static  # noqa: F401

pytestmark = pytest.mark.gpu
SCORINGS = [(1, -1, -1, 251), (1, -1, -1, 252), (6, -12, -6, 232), (7, -12, -6, 100),  # from the one
            (1, -2, -1, 1535), (127, -1, -1, 1409), (64, -128, -64, 1472), (3, -2, -125, 100),
            (1, -2, -1, 1536), (65, -128, -64, 100), (1, 0, -100, 1535)]  # to the other


@pytest.mark.parametrize("sc", SCORINGS, ids=lambda s: "_".join(map(str, s)))
def test_scorings(X, orc, sc):
    rng = np.random.default_rng(94)
    a, b, seeds = [], [], []
    for k in range(12):  # one read gains a base every 8
        t = rng.integers(0, 4, int(rng.integers(300, 1500))).astype(np.uint8)
        u = np.concatenate([np.append(t[q:q + 8], rng.integers(0, 4)) for q in range(0, len(t), 8)])
        u = u.astype(np.uint8)
        a.append(t if k % 2 else u)
        b.append(u if k % 2 else t)
        seeds.append((0, 0, 8))
    for w in (W.template_pairs(n_pairs=24, len_lo=300, len_hi=2000, seed=92),
              W.tiny_pairs(n_pairs=150, len_lo=0, len_hi=40, seed=93), W.from_sequences(a, b, seeds)):
        w.match, w.mismatch, w.gap, w.x = sc
        want = _oracle(orc, w)
        assert np.array_equal(_small(X, w)[0], want), (sc, w.name)
        assert np.array_equal(_static(X, w), want), (sc, w.name)


@pytest.mark.parametrize("sc", [(10, -9, -10, 400), (5, -4, -3, 600)], ids=lambda s: "_".join(map(str, s)))
def test_longest_extensions_of_a_larger_batch(X, orc, sc):
    w = W.uneven_pairs(n_pairs=4000, seed=95)
    w.match, w.mismatch, w.gap, w.x = sc
    assert np.array_equal(_small(X, w)[0], _oracle(orc, w))
