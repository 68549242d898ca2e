"""xdrop_align_static on a packed buffer of more than 2^31 words (no other call
takes one): its extensions then run on the scratch, which names bases in 64
bits, and those of a buffer just short of the limit on the windows."""
import numpy as np
import pytest

from paper_2309_07270_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("words", [2**31 - 2**22 - 1, 2**31 + 4096], ids=["last_packed", "beyond"])
def test_reads_at_the_end(orc, words):
    import torch

    from paper_2309_07270_gb300 import build
    from paper_2309_07270_gb300 import xdrop as X
    build.build()
    w = W.template_pairs(n_pairs=20, len_lo=500, len_hi=2500, seed=81)
    dev = X.DeviceInputs.from_workload(w)
    n = len(w.packed)
    buf = torch.empty(words, dtype=torch.int32, device="cuda:0")
    buf[:n] = dev.packed
    buf[-n:] = dev.packed
    off = dev.read_off.clone()
    half = len(off) // 2  # the later reads stand at the end of the buffer
    off[half:] += 16 * (words - n)
    for x in (20, 300, 900):  # 128 and 512 slots, the scratch
        X.xdrop_align_static(buf.data_ptr(), words, off.data_ptr(), dev.read_len.data_ptr(),
                             dev.read_len.numel(), dev.pairs.data_ptr(), dev.n_pairs,
                             X.scoring(1, -1, -1, x), int(w.read_len.max()), dev.out.data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        want = orc.align_pairs(w.packed, w.read_off, w.read_len, w.pairs, 1, -1, -1, x, nthreads=8)
        assert np.array_equal(dev.results().view(np.int32), want.view(np.int32)), x
