"""The warp-per-extension kernel against the oracle: small batches (which run
on it alone), the allocation-free call, and the extensions a narrower first
tier hands on."""
import numpy as np
import pytest

from paper_2309_07270_gb300 import workloads as W

pytestmark = pytest.mark.gpu
# the packed window's limits (x + 2 match + 2|gap| <= 255, match + |gap| <= 12), and beyond them
SCORINGS = [(1, -1, -1, 50), (1, -1, -1, 251), (1, -1, -1, 252), (6, -12, -6, 231), (7, -5, -6, 100),
            (2, -3, -2, 40), (1, 0, -1, 30), (11, -1, -1, 100), (1, -3, -1, 30), (7, -1, -2, 0)]


@pytest.fixture(scope="module")
def X():
    from paper_2309_07270_gb300 import build, xdrop
    build.build()
    return xdrop


def _oracle(orc, w):
    return orc.align_pairs(w.packed, w.read_off, w.read_len, w.pairs, w.match, w.mismatch, w.gap,
                           w.x, nthreads=8).view(np.int32)


def _sc(X, w):
    return X.scoring(w.match, w.mismatch, w.gap, w.x)


def _static(X, w):
    import torch
    d = X.DeviceInputs.from_workload(w)
    X.xdrop_align_static(d.packed.data_ptr(), d.packed.numel(), d.read_off.data_ptr(),
                         d.read_len.data_ptr(), d.read_len.numel(), d.pairs.data_ptr(), d.n_pairs,
                         _sc(X, w), int(max(w.read_len)), d.out.data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return d.results().view(np.int32)


def _small(X, w):
    with X.Aligner() as al:
        got = al.align(w.packed, w.read_off, w.read_len, w.pairs, _sc(X, w)).view(np.int32)
        return got, al.stats()


@pytest.mark.parametrize("sc", SCORINGS, ids=lambda s: "_".join(map(str, s)))
def test_scorings(X, orc, sc):
    for w in (W.template_pairs(n_pairs=30, len_lo=500, len_hi=2500, seed=61),
              W.tiny_pairs(n_pairs=200, len_lo=0, len_hi=40, seed=62)):  # around the block of 8 diagonals
        w.match, w.mismatch, w.gap, w.x = sc
        want = _oracle(orc, w)
        got, st = _small(X, w)
        assert st["tile_lanes"] == 32 and st["graph_replays"] == 0
        assert np.array_equal(got, want), (sc, w.name)
        assert np.array_equal(_static(X, w), want), (sc, w.name)


def test_drift_and_every_wider_tier(X, orc):
    rng = np.random.default_rng(63)
    a, b, seeds = [], [], []
    for k in range(24):
        t = rng.integers(0, 4, int(rng.integers(300, 2500))).astype(np.uint8)
        u = np.concatenate([np.append(t[q:q + 8], rng.integers(0, 4)) for q in range(0, len(t), 8)])
        a.append(t if k % 2 else u.astype(np.uint8))
        b.append(u.astype(np.uint8) if k % 2 else t)
        seeds.append((0, 0, 8))
    w = W.from_sequences(a, b, seeds, x=20)  # the window moves by hundreds of slots
    got, st = _small(X, w)
    assert np.array_equal(got, _oracle(orc, w)) and st["overflow_tasks"] == 0
    for x in (180, 700, 1500):  # past 128 slots, past 512
        wx = w.with_x(x)
        want = _oracle(orc, wx)
        got, st = _small(X, wx)
        assert np.array_equal(got, want), x
        assert st["overflow_tasks"] > 0 and (st["wide_tasks"] > 0) == (x > 180)
        assert np.array_equal(_static(X, wx), want), x


@pytest.mark.parametrize("n", [1, 608, 609])
def test_batch_sizes_around_the_switch(X, orc, n):
    """Up to 8 tasks per SM (608 pairs on 152 SMs) run here; more do not."""
    w = W.template_pairs(n_pairs=n, len_lo=30, len_hi=300, seed=64)
    got, _ = _small(X, w)
    assert np.array_equal(got, _oracle(orc, w))


def test_invalid_pairs_of_a_small_device_submit(X, orc):
    w = W.template_pairs(n_pairs=40, len_lo=300, len_hi=800, seed=65)
    want = _oracle(orc, w).reshape(-1, 7)
    bad = w.pairs.copy()
    bad[3]["seed_a"] = w.read_len[bad[3]["a"]]
    bad[7]["b"] |= X.XDROP_PAIR_RC  # no reverse complements in a device submit
    dev = X.DeviceInputs(w.packed, w.read_off, w.read_len, bad)
    with X.Aligner() as al:
        with pytest.raises(X.XdropError) as ei:
            al.align_device(dev, _sc(X, w))
    assert ei.value.code == X.XDROP_EINVAL
    got = dev.results().view(np.int32).reshape(-1, 7)
    assert (got[[3, 7]] == [0, 0, 0, 0, 0, 0, X.XDROP_STATUS_INVALID]).all()
    ok = np.setdiff1d(np.arange(40), [3, 7])
    assert np.array_equal(got[ok], want[ok])
