"""The library's host code over a CUDA runtime of host memory
(tests/fake_cuda.cpp): what a context does when a kernel reports an error, an
allocation fails or a result is late.  No kernel runs, so results are zeros."""
import ctypes
import importlib.util
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
PKG = os.path.join(os.path.dirname(HERE), "paper_2309_07270_gb300")


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    gxx = shutil.which("g++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if gxx is None or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    so = tmp_path_factory.mktemp("fake") / "libfake.so"
    subprocess.run([gxx, "-x", "c++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-pthread",
                    "-Wl,-Bsymbolic",  # not the CUDA runtime that torch has loaded
                    "-I", os.path.join(os.path.dirname(HERE), "include"), "-I", include, "-o",
                    str(so), os.path.join(HERE, "fake_cuda.cpp")], check=True)
    return str(so)


@pytest.fixture
def X(built, tmp_path):
    """The binding over a fresh copy of the fake library (4 SMs: 16 pairs and
    fewer are a small batch)."""
    so = shutil.copy(built, tmp_path / "libfake.so")
    spec = importlib.util.spec_from_file_location("xdrop_fake", os.path.join(PKG, "xdrop.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    mod.LIB_PATH = str(so)
    lib = mod.load()
    for name in ("fake_device_size", "fake_pool_reserved", "fake_seed_tables"):
        getattr(lib, name).argtypes = [ctypes.c_size_t]
        getattr(lib, name).restype = None
    lib.fake_device_used.restype = ctypes.c_size_t
    mod.fake = lib
    return mod


def _job(X, n, words=64):
    """n pairs of two 64-base reads in a buffer of `words` words."""
    pairs = np.zeros(n, X.PAIR_DTYPE)
    pairs["b"] = 1
    pairs["seed_len"] = 8
    off = np.array([0, 16 * words - 64], np.uint64)
    return np.zeros(words, np.uint32), off, np.array([64, 64], np.uint32), pairs


def test_a_lost_entry_is_reported_to_its_own_call(X):
    sc = X.scoring()
    with X.Aligner() as al:
        al.align(*_job(X, 40), sc)  # tuned
        X.fake.fake_lose_entries(1)
        with pytest.raises(X.XdropError) as ei:
            al.align(*_job(X, 40), sc)
        assert ei.value.code == X.XDROP_ECUDA and "never appeared" in str(ei.value)
        al.align(*_job(X, 40), sc)
        al.align(*_job(X, 4), sc)


def _long(X, length):
    """One pair of reads of `length` bases."""
    packed, off, lens, pairs = _job(X, 1, words=2 * (length // 16 + 1))
    off[1] = 16 * (length // 16 + 1)
    lens[:] = length
    return packed, off, lens, pairs


def test_a_failed_growth_leaves_no_stale_scratch(X):
    """The unbounded tier's buffer is freed before the larger one is asked for:
    when that fails, a later call must not run on the freed one."""
    sc = X.scoring()
    with X.Aligner() as al:
        al.align(*_long(X, 1000), sc)
        X.fake.fake_device_size(X.fake.fake_device_used() + 100_000)
        with pytest.raises(X.XdropError):
            al.align(*_long(X, 100_000), sc)
        al.align(*_long(X, 900), sc)
        assert X.fake.fake_bad_scratch() == 0


@pytest.mark.parametrize("budget", [0, 1 << 20], ids=["out_of_memory", "over_budget"])
def test_a_failed_load_leaves_no_half_read_set(X, budget):
    """Out of memory the old reads have gone with their buffer; a budget refuses
    before anything is freed, and they stay."""
    sc = X.scoring()
    packed, off, lens, pairs = _job(X, 3)
    out = np.zeros(3, X.RESULT_DTYPE)
    with X.Aligner(budget=budget) as al:
        X.xdrop_load_reads(al.ctx, packed, off, lens)
        X.fake.fake_device_size(X.fake.fake_device_used() + 100_000)
        with pytest.raises(X.XdropError):
            X.xdrop_load_reads(al.ctx, *_job(X, 3, words=1 << 20)[:3])
        if budget:
            X.xdrop_sync(al.ctx, X.xdrop_submit_pairs(al.ctx, pairs, sc, out))
        else:
            with pytest.raises(X.XdropError) as ei:
                X.xdrop_submit_pairs(al.ctx, pairs, sc, out)
            assert ei.value.code == X.XDROP_EINVAL


def _device_submit(X, al, job, sc):
    packed, off, lens, pairs = job
    out = np.zeros(len(pairs), X.RESULT_DTYPE)
    p = [a.ctypes.data for a in (packed, off, lens, pairs, out)]
    t = X.xdrop_submit_device(al.ctx, p[0], len(packed), p[1], p[2], len(lens), p[3], len(pairs),
                              sc, p[4])
    return t, (job, out)


@pytest.mark.parametrize("call", ["submit", "load_reads", "scratch", "seeds"])
def test_kept_memory_makes_room_for_a_call(X, call):
    """Idle tickets keep their buffers and seed discovery its pages; a call that
    runs out of memory gets them, as it did when nothing was kept."""
    sc, mb = X.scoring(), 1 << 20
    with X.Aligner() as al:
        X.xdrop_load_reads(al.ctx, *_job(X, 3)[:3])
        al.align(*_job(X, 4, words=16 * mb // 4), sc)  # a ticket with 16 MB stays
        X.xdrop_find_candidates(al.ctx, k=9)           # makes the pool
        X.fake.fake_pool_reserved(16 * mb)
        X.fake.fake_device_size(X.fake.fake_device_used() + 2 * mb)
        if call == "submit":
            al.align(*_job(X, 4, words=24 * mb // 4), sc)
        elif call == "load_reads":
            X.xdrop_load_reads(al.ctx, *_job(X, 3, words=12 * mb // 4)[:3])
        elif call == "scratch":
            t, _keep = _device_submit(X, al, _long(X, 300_000), sc)
            X.xdrop_sync(al.ctx, t)
        else:
            X.fake.fake_seed_tables(24 * mb)
            X.xdrop_find_candidates(al.ctx, k=11)
        assert X.fake.fake_device_used() <= 35 * mb


def test_a_device_submit_leaves_the_large_buffers_idle(X):
    """It needs none; the next host submit finds its buffer kept."""
    sc = X.scoring()
    with X.Aligner() as al:
        big = _job(X, 4, words=1 << 20)
        packed, off, lens, pairs = big
        out = [np.zeros(4, X.RESULT_DTYPE) for _ in range(2)]
        small = _job(X, 4)
        t = [X.xdrop_submit(al.ctx, *job, sc, o) for job, o in zip((big, small), out)]
        for k in t:
            X.xdrop_sync(al.ctx, k)
        used = X.fake.fake_device_used()
        t, _keep = _device_submit(X, al, _job(X, 4), sc)
        al.align(*big, sc)
        assert X.fake.fake_device_used() == used
        X.xdrop_sync(al.ctx, t)


@pytest.mark.parametrize("order", [(1, 0, 1), (0, 1, 0)], ids=["tuned_first", "forced_first"])
def test_a_forced_tile_runs_without_the_longest_cut(X, order):
    """The longest tasks skip the first tile only when it was tuned: the captured
    launch of the one must not be replayed for the other."""
    sc = X.scoring()
    with X.Aligner() as al:
        al.align(*_job(X, 40), sc)
        lanes, cells = al.tile()
        for tuned in order:
            al.set_tile(*((0, 0) if tuned else (lanes, cells)))
            al.align(*_job(X, 40), sc)
            assert X.fake.fake_last_longest() == tuned


def test_device_bytes_holds_the_seed_pool(X):
    """device_bytes is what the context holds now, pages kept between calls too."""
    with X.Aligner() as al:
        X.xdrop_load_reads(al.ctx, *_job(X, 3)[:3])
        before = al.stats()["device_bytes"]
        X.xdrop_find_candidates(al.ctx, k=9)
        X.fake.fake_pool_reserved(1 << 20)
        assert al.stats()["device_bytes"] == before + (1 << 20)


def test_one_thread_polls(X):
    """Waiting threads beside the first sleep until their result is there."""
    import threading
    sc = X.scoring()
    X.fake.fake_late_us(1500)
    with X.Aligner() as al:
        job = _job(X, 4)
        out = [np.zeros(4, X.RESULT_DTYPE) for _ in range(6)]
        tickets = [X.xdrop_submit(al.ctx, *job, sc, o) for o in out]
        X.fake.fake_polling_max()
        th = [threading.Thread(target=X.xdrop_sync, args=(al.ctx, t)) for t in tickets]
        for t in th:
            t.start()
        for t in th:
            t.join()
        assert X.fake.fake_polling_max() == 1
