"""Scorings in which a mismatch costs more than two gaps run as if it cost
two (packed where that fits 16 bits): the oracle's results, through every
call, and the limits of the scoring as given."""
import numpy as np
import pytest

from paper_2309_07270_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def X():
    from paper_2309_07270_gb300 import build, xdrop
    build.build()
    return xdrop


@pytest.mark.parametrize("sc", [(2, -3, -1, 30), (1, -3, -1, 50), (1, -129, -1, 10), (1, -9000, -1, 40),
                                (3, -500, -100, 300), (1, -40, -1, 1100)],
                         ids=lambda s: "_".join(map(str, s)))
def test_matches_oracle(X, orc, sc):
    s = X.scoring(*sc)
    for w in (W.template_pairs(n_pairs=700, len_lo=100, len_hi=600, seed=81),
              W.template_pairs(n_pairs=30, len_lo=500, len_hi=1500, seed=82),
              W.tiny_pairs(n_pairs=900, seed=83)):
        want = orc.align_pairs(w.packed, w.read_off, w.read_len, w.pairs, *sc, nthreads=8).view(np.int32)
        for mode in (X.XDROP_MODE_BATCHED, X.XDROP_MODE_PLAIN):
            with X.Aligner(mode=mode) as al:
                got = al.align(w.packed, w.read_off, w.read_len, w.pairs, s).view(np.int32)
                assert np.array_equal(got, want), (sc, w.name, mode)
        with X.Aligner() as al:
            al.set_tile(8, 8)
            got = al.align(w.packed, w.read_off, w.read_len, w.pairs, s).view(np.int32)
            assert np.array_equal(got, want), (sc, w.name)


@pytest.mark.parametrize("n", [40, 900])
def test_limits_are_those_of_the_scoring_as_given(X, n):
    """|mismatch| (len_a + len_b) < 2^25 decides, not two gaps."""
    w = W.template_pairs(n_pairs=n, len_lo=100, len_hi=300, seed=84)
    tot = w.read_len[w.pairs["a"]].astype(np.int64) + w.read_len[w.pairs["b"]]
    mis = -int((1 << 25) // int(np.median(tot)))
    bad = -mis * tot >= 1 << 25
    assert bad.any() and not bad.all()
    dev = X.DeviceInputs.from_workload(w)
    for tile in (None, (8, 8)):
        with X.Aligner() as al:
            if tile:
                al.set_tile(*tile)
            with pytest.raises(X.XdropError):
                al.align_device(dev, X.scoring(1, mis, -1, 20))
        assert np.array_equal(dev.results()["status"] == X.XDROP_STATUS_INVALID, bad)
