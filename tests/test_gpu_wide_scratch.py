"""The unbounded tier's scratch follows the reads of every call: contexts that
meet longer reads than before, on bands wider than 512 slots, against the
oracle."""
import numpy as np
import pytest

from paper_2309_07270_gb300 import workloads as W

pytestmark = pytest.mark.gpu
X_DROP = 1200  # identical reads: the band holds most of the rectangle


@pytest.fixture(scope="module")
def X():
    from paper_2309_07270_gb300 import build, xdrop
    build.build()
    return xdrop


def _reads(n, length, seed):
    """n pairs of copies of one read, seeded at their start (the right
    extension is everything)."""
    t = np.random.default_rng(seed).integers(0, 4, length).astype(np.uint8)
    return W.from_sequences([t] * n, [t] * n, [(0, 0, 8)] * n, x=X_DROP)


def _want(orc, w):
    one = orc.align_pairs(w.packed, w.read_off, w.read_len, w.pairs[:1], 1, -1, -1, X_DROP)
    return np.tile(one.view(np.int32), len(w.pairs))


@pytest.mark.parametrize("n", [3, 700])  # a small batch, and one replayed from a graph
def test_growing_reads(X, orc, n):
    """The second growth leaves room for the third without a new buffer."""
    sc = X.scoring(1, -1, -1, X_DROP)
    with X.Aligner() as al:
        for length in (1000, 1100, 1400):
            w = _reads(n, length, length)
            got = al.align(w.packed, w.read_off, w.read_len, w.pairs, sc).view(np.int32)
            assert al.stats()["wide_tasks"] > 0
            assert np.array_equal(got, _want(orc, w)), length


@pytest.mark.parametrize("n,short,long", [(3, 600, 1500), (700, 600, 1500), (3, 40, 15000)],
                         ids=["small", "graph", "longer_than_the_scratch"])
@pytest.mark.parametrize("tile", [None, (2, 32 | 0x100)], ids=["tuned", "forced"])
def test_read_lengths_rewritten_in_place(X, orc, n, short, long, tile):
    """The arrays of a device submit may hold longer reads once its ticket is
    synced: first the reads' heads, then the whole reads, at the same addresses."""
    w = _reads(n, long, long)
    sc = X.scoring(1, -1, -1, X_DROP)
    dev = X.DeviceInputs.from_workload(w)
    whole = dev.read_len.clone()
    with X.Aligner() as al:
        if tile:
            al.set_tile(*tile)
        dev.read_len.fill_(short)
        al.align_device(dev, sc)
        dev.read_len.copy_(whole)
        dev.out.fill_(-1)
        for _ in range(2):  # the first finds the slices too short
            al.align_device(dev, sc)
            assert al.stats()["wide_tasks"] > 0
            assert np.array_equal(dev.results().view(np.int32), _want(orc, w))
