"""The host side of the tensor-core kernels on a CUDA runtime of host functions (tests/launch_on_fake_cuda.cpp): a driver that hands
out no tensor maps is no reason to refuse a call (every tile is then gathered row by row); the row dots' grid; the backward's
workspace.  No GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_04312_b200", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    so = str(tmp_path_factory.mktemp("launch") / "launch.so")
    # device code as PTX only: none of it is run
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=compute_100a", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-Xlinker", "-Bsymbolic", "-cudart", "none", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-o", so,
                    os.path.join(CSRC, "mate_fwd_tc.cu"), os.path.join(CSRC, "mate_bwd_tc.cu"),
                    os.path.join(ROOT, "tests", "launch_on_fake_cuda.cpp")], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("backward,launches", [(0, 1), (1, 2)])
def test_calls_go_through_without_maps(lib, backward, launches):
    n, bulk = ctypes.c_int(), ctypes.c_int()
    assert lib.call(backward, ctypes.byref(n), ctypes.byref(bulk)) == 0
    assert (n.value, bulk.value) == (launches, 0)


@pytest.mark.parametrize("n_ctas", [132, 148])
def test_row_dots_go_in_one_wave_with_as_few_rows_per_thread_as_can_be(lib, n_ctas):
    # blocks of 32 or 64 rows where eight of them to an SM are enough, of 128 for more
    one, two = n_ctas * 8 * 32, n_ctas * 8 * 64
    for rows, per_block in ((1, 32), (n_ctas * 6 * 32 + 1, 32), (one, 32), (one + 1, 64), (n_ctas * 6 * 64 + 1, 64), (two, 64), (two + 1, 128)):
        assert lib.rowdot_grid(1, rows, n_ctas) == -(-rows // per_block), rows


@pytest.mark.parametrize("B,H,N,T", [(1, 12, 8192, 0), (4, 12, 2047, 0), (64, 12, 8192, 8192 + 63 * 128), (3, 1, 5, 7)])
def test_backward_workspace_goes_by_rows_of_the_tensors(lib, B, H, N, T):
    # 40 bytes a row; one long example among short ones does not make a packed batch as long as so many of them
    lib.backward_workspace.restype = ctypes.c_size_t
    rows = H * T if T else B * H * N
    assert 40 * rows <= lib.backward_workspace(B, H, N, T) <= 40 * rows + 1024
