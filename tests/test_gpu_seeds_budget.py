"""Seed discovery under a device memory budget: reads that share nothing need no
room for partners."""
import numpy as np
import pytest

from test_gpu_seeds import X, pack  # noqa: F401

pytestmark = pytest.mark.gpu


def test_no_reliable_kmer_needs_no_partner_tables(X):
    """20,000 reads of 40 bases: tables of 20 MB, and 82 MB for partners that a
    window above every count does not ask for."""
    rng = np.random.default_rng(14)
    packed, off, lens = pack(list(rng.integers(0, 4, (20_000, 40)).astype(np.uint8)))
    with X.Aligner(budget=64 << 20) as al:
        X.xdrop_load_reads(al.ctx, packed, off, lens)
        pairs, shared = X.xdrop_find_candidates(al.ctx, 9, 900, 1000)
        assert len(pairs) == len(shared) == 0
        st = X.xdrop_get_seed_stats(al.ctx)
        assert st["runs"] > 0 and st["nonzeros"] == 0 and st["product"] == X.XDROP_SEEDS_ROWWISE
        with pytest.raises(X.XdropError) as ei:  # shared k-mers do
            X.xdrop_find_candidates(al.ctx, 9, 1, 1000)
        assert ei.value.code == X.XDROP_ENOMEM
