"""The C-ABI library loads and exports every function that include/mate.h declares (no GPU)."""
import ctypes
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    with open(os.path.join(ROOT, "include", "mate.h")) as f:
        text = f.read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(mate_[a-z_0-9]+)\s*\(", text)))


@pytest.fixture(scope="module")
def lib():
    from paper_2109_04312_b200 import build
    return ctypes.CDLL(build.build())


def test_header_declares_the_three_calls():
    names = declared_functions()
    for need in ("mate_plan", "mate_attn_fwd", "mate_attn_bwd"):
        assert need in names


def test_library_exports_every_declared_symbol(lib):
    for name in declared_functions():
        assert hasattr(lib, name), name


def test_status_strings(lib):
    lib.mate_status_string.restype = ctypes.c_char_p
    seen = set()
    for s in range(0, -8, -1):
        msg = lib.mate_status_string(s).decode()
        assert msg and msg != "unknown status"
        seen.add(msg)
    assert len(seen) == 8
    assert lib.mate_status_string(-99).decode() == "unknown status"


def test_null_arguments_are_rejected_without_a_gpu(lib):
    # argument checks come before any CUDA call, so they work on a machine without a device
    out = ctypes.c_void_p()
    assert lib.mate_plan(None, None, 1, 8, 0, None, 1, 1, 1, None, ctypes.byref(out)) == -1
    assert lib.mate_plan_get(None, 0, None, None, None) == -1
    assert lib.mate_plan_useful_pairs(None, None) == -1
    assert lib.mate_plan_destroy(None) == 0
    f = ctypes.c_size_t()
    assert lib.mate_attn_workspace_bytes(None, 64, 0, 0, ctypes.byref(f), ctypes.byref(f)) == -1


@pytest.mark.parametrize("H", [1 << 20, 1 << 28, (1 << 29) + 1])
def test_number_of_heads_is_no_reason_to_refuse(lib, H):
    # the check of the views comes last: a bad one at the end says that nothing else was refused
    views = (ctypes.c_uint8 * H)()
    views[H - 1] = 2
    ids, out = (ctypes.c_int32 * 1)(), ctypes.c_void_p()
    assert lib.mate_plan(ids, ids, 1, 1, 0, views, H, 1, 1, None, ctypes.byref(out)) == -1


def test_binding_fails_loudly_without_the_library(monkeypatch):
    from paper_2109_04312_b200 import api
    monkeypatch.setattr(api, "_lib", None)
    monkeypatch.setattr(api, "_LIB_PATH", os.path.join(ROOT, "no_such_dir", "libmate.so"))
    with pytest.raises(ImportError):
        api._load()


def test_memory_that_is_not_to_be_had_is_a_status(lib):
    # lists as long as the (absurd) inputs do not fit the process's address space: in the entry point, and in the plan
    code = """
import ctypes, mmap, resource, sys
lib = ctypes.CDLL(sys.argv[1])
held = int(open("/proc/self/statm").read().split()[0]) * mmap.PAGESIZE
buf = (ctypes.c_ubyte * 64)()
out = ctypes.c_void_p()
arg = lambda x: ctypes.c_void_p(ctypes.addressof(x))
B = 1 << 26
zeros = mmap.mmap(-1, 4 * B, prot=mmap.PROT_READ | mmap.PROT_WRITE)
prefix = (ctypes.c_ubyte * 1).from_buffer(zeros)
resource.setrlimit(resource.RLIMIT_AS, (held + 4 * B + (128 << 20), resource.RLIM_INFINITY))
big = 2 ** 31 - 1
rc = [lib.mate_plan(arg(buf), arg(buf), big, 1, 0, arg(buf), 1, 1, 1, None, ctypes.byref(out)),
      lib.mate_plan_sat(arg(buf), arg(buf), big, 1, 0, 1, 1, 1, None, ctypes.byref(out)),
      lib.mate_plan_packed(arg(buf), arg(buf), B, arg(prefix), arg(prefix), arg(buf), 1, 1, 1, None, ctypes.byref(out)),
      lib.mate_plan_varlen(arg(buf), arg(buf), B, 1, arg(prefix), arg(buf), 1, 1, 1, 0, None, ctypes.byref(out))]
print(rc, out.value)
"""
    r = subprocess.run([sys.executable, "-c", code, lib._name], capture_output=True, text=True)
    assert (r.returncode, r.stdout.strip()) == (0, "[-6, -6, -6, -6] None"), r.stderr
