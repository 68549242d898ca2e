"""Columns of the row-wise product at the sizes its kernels split at: 16
members a half warp reads at once, 32 run entries a warp takes at once,
with k-mers that repeat inside a read across those edges."""
import numpy as np
import pytest

from oracle import seeds as S

from test_gpu_seeds import X, gpu, pack, same  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 15, 16, 17, 18, 31, 32, 33, 34, 65, 300])
@pytest.mark.parametrize("repeats", [1, 3])
def test_column_sizes(X, n, repeats):
    rng = np.random.default_rng(100 * n + repeats)
    core = rng.integers(0, 4, 40).astype(np.uint8)
    reads = []
    for _ in range(n):  # each: the core, `repeats` times, between random ends
        parts = [rng.integers(0, 4, int(rng.integers(0, 30))).astype(np.uint8)]
        for _ in range(repeats):
            parts += [core, rng.integers(0, 4, int(rng.integers(0, 9))).astype(np.uint8)]
        r = np.concatenate(parts)
        reads.append(r if rng.random() < 0.5 else (3 - r[::-1]).astype(np.uint8))
    reads.insert(int(rng.integers(0, n)), np.zeros(0, np.uint8))
    packed, off, lens = pack(reads)
    for lo, hi in ((1, 1024), (n * repeats, n * repeats), (n * repeats + 1, 1024)):
        want = S.candidate_pairs(packed, off, lens, k=15, lo=lo, hi=hi)
        same(gpu(X, packed, off, lens, 15, lo, hi, rowwise=True), want)
