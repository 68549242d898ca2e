"""CPU check of the packed band kernel's relative frame against the oracle.

The bit-level model (``relative16_model``) must reach the oracle's result
exactly whenever the band fits the window, over scorings at the edges of
the range, with no half that wraps or carries; and the host-side rules of
the kernel header must equal the model's over a grid that crosses every
limit.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

import packed16_model as P
import relative16_model as R
from paper_2309_07270_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SCORINGS = [
    (1, -1, -1, 50), (1, 0, -1, 20), (2, -3, -2, 30), (1, -2, -1, 100),
    (64, -128, -64, 1472), (64, -128, -64, 767),  # largest of 16- and of 32-slot lanes
    (3, -2, -125, 100), (127, -1, -1, 1409), (127, -1, -1, 767),
    (1, -2, -1, 1535), (1, -2, -1, 1019), (1, -2, -1, 507), (32, -64, -32, 383), (7, -1, -2, 0), (4, -4, -3, 40),
]


def cases(seed, n, slots):
    rng = np.random.default_rng(seed)
    scorings = [sc for sc in SCORINGS if R.relative_ok(*sc, slots)]
    for k in range(n):
        la, lb = int(rng.integers(0, 260)), int(rng.integers(0, 260))
        t = rng.integers(0, 4, max(la, lb) + 40).astype(np.uint8)
        b = (W.mutate(t, rng)[0], rng.integers(0, 4, lb).astype(np.uint8), t)[k % 3]
        yield scorings[(k // 3) % len(scorings)], t[:la], b[:lb]


@pytest.mark.parametrize("lanes,regs", [(4, 4), (4, 8), (2, 16), (4, 16), (32, 2), (1, 16), (1, 32), (2, 32)])
def test_model_matches_oracle(orc, lanes, regs):
    done = 0
    for sc, a, b in cases(lanes * regs, 42, 2 * regs):
        got = R.extend(a, b, *sc, lanes=lanes, regs=regs)
        if not got[3]:
            assert tuple(got[:3]) == tuple(orc.extend(a, b, *sc)[:3]), (sc, len(a), len(b))
            done += 1
    assert done >= 14


@pytest.mark.parametrize("lanes,regs", [(4, 8), (2, 16)])
@pytest.mark.parametrize("sc", [(1, -1, -1, 50), (127, -1, -1, 700), (64, -128, -64, 700)])
def test_long_reads_sink_and_lift_pruned_slots(orc, lanes, regs, sc):
    """1,500 identical bases raise the threshold by the most it can rise per
    diagonal, so pruned slots sink fastest: none may wrap before a lift."""
    t = np.random.default_rng(9).integers(0, 4, 1500).astype(np.uint8)
    st = {}
    got = R.extend(t, t, *sc, lanes=lanes, regs=regs, stats=st)
    assert not got[3] and tuple(got[:3]) == tuple(orc.extend(t, t, *sc)[:3])
    assert st["lift"] >= 1500 // R.lift_period(sc[0], sc[2], 2 * regs) - 1


@pytest.mark.parametrize("lanes,regs", [(4, 8), (2, 16), (1, 32), (16, 2)])
def test_drifting_band_shifts_the_window(orc, lanes, regs):
    rng = np.random.default_rng(17)
    t = rng.integers(0, 4, 480).astype(np.uint8)
    d = np.concatenate([np.append(t[k:k + 8], rng.integers(0, 4)) for k in range(0, 480, 8)])
    shifted = {}
    for a, b in [(t, d), (d, t)]:
        got = R.extend(a, b, 1, -1, -1, 20, lanes=lanes, regs=regs, stats=shifted)
        assert not got[3] and tuple(got[:3]) == tuple(orc.extend(a, b, 1, -1, -1, 20)[:3])
    assert shifted["up"] >= 4 and shifted["down"] >= 4


PROGRAM = r"""
#include <stdio.h>
#include "xd_lockstep16.cuh"
int main(void)
{
    const int match[] = {1, 2, 3, 7, 64, 127, 128}, gap[] = {-1, -2, -3, -64, -127, -128};
    const int mis[] = {0, -1, -2, -3, -4, -127, -128, -129};
    const int x[] = {0, 1, 50, 505, 506, 507, 765, 766, 767, 1017, 1018, 1019, 1020, 1535, 1536};
    for (int a : match) for (int g : gap) for (int b : mis) for (int c : x) {
        const xd::Scoring sc{a, b, g, c};
        if (!xd::packed16_ok(sc)) continue;
        printf("%d %d %d %d %d %d %d %d %d %d\n", a, b, g, c, (int)xd::relative_ok<16>(sc),
               (int)xd::relative_ok<32>(sc), (int)xd::relative_ok<64>(sc),
               (int)xd::subst_folds(sc), xd::lift_period<16>(sc), xd::lift_period<32>(sc));
    }
    return 0;
}
"""


def test_kernel_rules_equal_the_model(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "rules.cu", tmp_path / "rules"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_2309_07270_gb300", "csrc"), "-I",
                    os.path.join(ROOT, "include"), "-o", str(exe), str(src)], check=True)
    rows = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    n = 0
    for m, mis, g, x, ok16, ok32, ok64, folds, p16, p32 in (map(int, r.split()) for r in
                                                      rows.splitlines()):
        assert bool(ok16) == R.relative_ok(m, mis, g, x, 16) and ok16  # every packed scoring
        assert bool(ok32) == R.relative_ok(m, mis, g, x, 32)
        assert not ok32 or P.fits(m, mis, g, x, 32)
        assert bool(ok64) == R.relative_ok(m, mis, g, x, 64)
        assert bool(folds) == R.subst_folds(m, mis, g)
        assert (p16, p32) == (R.lift_period(m, g, 16), R.lift_period(m, g, 32))
        n += 1
    assert n > 500
