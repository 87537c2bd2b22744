"""Mixed pair-once kernels below 65,536 bodies, on the CPU: the block choice
(csrc/pair_once_plan.h through tests/msym_plan_shim.cpp) and the schedule of
the 128-entry block kernel (csrc/sym_mixed.cu).

The choice, on 152 SMs: every ordered pair below 2,048 bodies, 128-entry blocks
while the block pairs fill 608 CTAs at most once (4,352 bodies) or at least
five times (9,857 bodies) and the rows stay in the L2 cache, 512-entry blocks
above (20,992 bodies), none from 65,536 bodies (the other function's).

The schedule: an emulation of a CTA's index arithmetic -- warp w takes the 16
rotation steps from 16 (w & 1) of chunk w >> 1, lane l at step k meets its
four targets 32 a + l with the two entries of pair block (l + k) mod 32 --
must meet every (target, source) of an off-diagonal item once and every
unordered pair of a diagonal one once, and hand each reaction sum back as the
sum of the pair block that the kernel files it under."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2112_15079_gb300", "csrc")


@pytest.fixture(scope="module")
def block(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = str(tmp_path_factory.mktemp("ms") / "libms.so")
    subprocess.run([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, os.path.join(HERE, "msym_plan_shim.cpp"),
                    "-o", out], check=True)
    lib = ctypes.CDLL(out)

    def f(sizes, nsm=152):
        a = np.ascontiguousarray(sizes, dtype=np.int64)
        return lib.ms_block(a.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(a.size), ctypes.c_int64(nsm))
    return f


@pytest.mark.parametrize("n,want", [(1, 0), (2047, 0), (2048, 128), (4352, 128), (4353, 0), (8192, 0), (9856, 0),
                                    (9857, 128), (10425, 128), (20480, 128), (20992, 512), (65535, 512), (65536, 0),
                                    (1048576, 0)])
def test_single_system(block, n, want):
    assert block([n]) == want


def test_batches(block):
    assert block([200] * 20000) == 128      # few rows each, however many bodies
    assert block([31] * 1000) == 0          # one round and a half of single blocks
    assert block([1500]) == 0 and block([1500] * 64) == 128
    assert block([5000] * 10) == 128
    assert block([5000] * 100) == 512       # the rows leave the cache
    rng = np.random.default_rng(0)
    assert block(rng.integers(1000, 20001, 64)) == 512
    assert block([300, 70000]) == 0         # a large system: the other function's
    assert block([65535] * 4000) == 0       # rows beyond the memory bound


@pytest.mark.parametrize("diag", [False, True])
def test_schedule(diag):
    met = np.zeros((128, 128), int)
    for w in range(4):
        chunk, k0 = w >> 1, 16 * (w & 1)
        held = np.arange(32)  # the pair block whose sums lane l holds, less the steps taken
        for k in range(k0, k0 + 16):
            for lane in range(32):
                m = (lane + k) & 31
                if k == k0:
                    held[lane] = m
                assert held[lane] == m
                for a in range(4):
                    for h in range(2):
                        t, f = 32 * a + lane, 64 * chunk + 2 * m + h
                        met[t, f] += (not diag) or t < f
            held = np.roll(held, -1)  # every lane takes the sums of the lane above
        assert np.array_equal(held, (np.arange(32) + k0 + 16) & 31)
    assert np.array_equal(met, np.triu(np.ones((128, 128), int), 1) if diag else np.ones((128, 128), int))
