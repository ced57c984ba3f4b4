"""The plan by which a block of the path kernels hands its batches to its warps
(csrc/simr_items.h), compiled for the host: the items cover the block's batches, their
rows fit the shared memory, and no warp is left with much more than its share.
"""
import ctypes
import heapq
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("items") / "items_test")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2402_12111_gb300", "csrc"), "-o", so,
                    os.path.join(ROOT, "tests", "c", "item_plan.cpp")], check=True)
    lib = ctypes.CDLL(so)
    u64, vp = ctypes.c_uint64, ctypes.c_void_p
    lib.plan.argtypes = [u64, u64, ctypes.c_int, u64, u64, vp, vp]
    lib.items.argtypes = [vp, u64, vp, ctypes.c_int64]
    lib.items.restype = ctypes.c_int64
    lib.plan_size.restype = u64
    return lib


ITEM_BYTES = 208 * 1024


def _plan(lib, batches, grid, warps, row, bytes_):
    I = ctypes.create_string_buffer(lib.plan_size())
    facts = (ctypes.c_uint64 * 4)()
    lib.plan(batches, grid, warps, row, bytes_, I, facts)
    return I, dict(zip(("warps", "bytes", "rows", "levels"), (int(x) for x in facts)))


def _ends(lib, I, nb):
    ends = np.zeros(1 << 16, np.uint64)
    n = lib.items(I, nb, ends.ctypes.data, ends.size)
    return None if n < 0 else ends[:n].astype(np.int64)


def _makespan(sizes, warps):
    """Time of the last warp when each takes the next item as it gets free, a unit per batch."""
    free = [0] * warps
    for s in sizes:
        heapq.heappush(free, heapq.heappop(free) + int(s))
    return max(free)


# (sums a strike, most warps, bytes taken before the rows per strike and in all): pricing,
# 3, 5 and 11 scenarios, adjoint QE and QE-M, basket of 8
KERNELS = [(2, 24, 16, 0), (2, 32, 16, 4096), (4, 20, 16, 832), (7, 24, 16, 832), (9, 16, 16, 0), (9, 24, 16, 8224),
           (9, 28, 16, 2048), (2, 20, 4, 0)]


@pytest.mark.parametrize("sums,warps,per_strike,other", KERNELS)
@pytest.mark.parametrize("strikes", [1, 32, 64, 96, 128, 160, 224, 256, 512, 1024])
def test_plans_cover_fit_and_balance(lib, sums, warps, per_strike, other, strikes):
    if strikes > (1024 if sums == 2 else 256):
        pytest.skip("past the entry points' strike limit")
    row, bytes_ = sums * strikes, ITEM_BYTES - 16 - per_strike * strikes - other
    rng = np.random.default_rng(strikes * 100 + sums)
    grid = 152
    sizes = list(range(1, 70)) + [108, 109, 216] + [int(x) for x in np.exp(rng.uniform(np.log(70), np.log(40000), 40))]
    for most in sizes:
        for batches in (grid * most, grid * most - 1) + ((grid * (most - 1) + 1,) if most > 1 else ()):
            I, f = _plan(lib, batches, grid, warps, row, bytes_)
            assert 1 <= f["warps"] <= warps and f["bytes"] <= bytes_ + 8, (most, f)
            for nb in {batches // grid, most} - {0}:
                ends = _ends(lib, I, nb)
                assert ends is not None and len(ends) <= f["rows"], (most, nb, f)
                # the launch ends with its fullest blocks, whose whole batches cannot end
                # before ceil(most / warps); a sixteenth more is allowed for items that are
                # several batches long
                got = _makespan(np.diff(ends, prepend=0), f["warps"])
                assert got <= -(-most // f["warps"]) * 17 // 16, (most, nb, f, got)


def test_grid_smaller_than_the_device(lib):
    for batches in (1, 2, 151):
        I, f = _plan(lib, batches, batches, 24, 64, ITEM_BYTES - 1024)
        assert f["warps"] == 1 and list(_ends(lib, I, 1)) == [1]
