"""The claims on the overflow list (csrc/xd_claim.cuh) on the CPU, one memory
operation at a time in random order with threads held up for hundreds of
operations: no position past the entries, none twice, none without an owner."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    so = tmp_path_factory.mktemp("claim_emu") / "libclaim_emu.so"
    subprocess.run([gxx, "-O2", "-std=c++17", "-Wall", "-Werror", "-pthread", "-shared", "-fPIC",
                    "-o", str(so), os.path.join(HERE, "claim_emulator.cpp")], check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("threads,each", [(1, 5), (2, 8), (5, 4), (8, 6)])
def test_every_entry_has_one_owner(lib, threads, each):
    for seed in range(40):
        assert lib.emulate_claims(threads, each, seed) == 0, seed
