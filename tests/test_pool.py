"""The pool behind the plans' memory, on a CUDA runtime of host functions (tests/fake_cuda_runtime.cpp): what it
does when a call fails, and when it waits.  No GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_04312_b200", "csrc")


@pytest.fixture
def pool(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    so = str(tmp_path / "pool.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(cuda, "include"), "-x", "c++", os.path.join(CSRC, "mate_pool.cu"),
                    os.path.join(ROOT, "tests", "fake_cuda_runtime.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    for name in ("pool_take", "pool_give", "plan_waits"):
        getattr(lib, name).argtypes = {"pool_take": [ctypes.c_int, ctypes.c_size_t, ctypes.c_size_t],
                                       "pool_give": [ctypes.c_int, ctypes.c_size_t],
                                       "plan_waits": [ctypes.c_size_t, ctypes.c_size_t]}[name]
    return lib


def test_blocks_are_reused_and_bounded(pool):
    for i in range(20):
        assert pool.pool_take(i, 100000, 1)
    for i in range(20):
        pool.pool_give(i, 1)
    assert pool.fake_live() == 16                     # the others have been freed
    assert pool.pool_take(0, 100000, 1) and pool.fake_device_syncs() == 0    # behind its last use on the stream
    assert pool.pool_take(1, 100000, 2) and pool.fake_device_syncs() == 1    # last used on another stream
    pool.pool_give(1, 0)
    assert pool.pool_take(2, 100000, 0) and pool.fake_device_syncs() == 2    # two unknown streams are not one
    assert pool.fake_live() == 16 and pool.fake_bad_frees() == 0


def test_a_block_whose_wait_fails_is_gone(pool):
    assert pool.pool_take(0, 100000, 1)
    pool.pool_give(0, 1)
    pool.fake_fail_device_sync(1)
    assert not pool.pool_take(1, 100000, 2)
    assert not pool.pool_holds(1)
    pool.pool_give(1, 2)                              # what mate_plan_destroy does with a plan that was not finished
    pool.fake_fail_device_sync(0)
    for i in (2, 3):
        assert pool.pool_take(i, 100000, 2) and pool.pool_is_live(i)
    for i in (2, 3):
        pool.pool_give(i, 2)
    assert pool.fake_bad_frees() == 0


def test_a_plan_is_waited_for_on_any_stream_but_its_own(pool):
    assert pool.plan_waits(1, 1) == 0
    assert pool.plan_waits(1, 2) == 1
    assert pool.plan_waits(0, 1) == 1 and pool.plan_waits(1, 0) == 1
    assert pool.plan_waits(0, 0) == 1                 # two unknown streams are not one
