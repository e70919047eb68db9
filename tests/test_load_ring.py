"""The barriers between the loader warps of the tensor-core kernels and the readers of what they load (csrc/load_ring.h), as a
model on the CPU (tests/load_ring_model.cpp): no wait passes before the phase it is for is over, whatever
the order in which the roles get on, and no run stands still."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("model") / "model.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2109_04312_b200", "csrc"),
                    os.path.join(ROOT, "tests", "load_ring_model.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def early_and_stuck(fn, bwd, runs, most, seed):
    out = (ctypes.c_int * 2)()
    fn(int(bwd), runs, most, seed, out)
    return out[0], out[1]


@pytest.mark.parametrize("kernel", ["forward", "backward"])
@pytest.mark.parametrize("most", [1, 2, 4, 12])  # tiles of an item; items without a tile are always among them
def test_no_wait_passes_early(model, kernel, most):
    assert early_and_stuck(model.as_built, kernel == "backward", 2500, most, 7 + most) == (0, 0)


@pytest.mark.parametrize("kernel", ["forward", "backward"])
def test_one_barrier_per_buffer_is_not_enough_for_teams(model, kernel):
    early, _ = early_and_stuck(model.teams, kernel == "backward", 2500, 2, 11)
    assert early > 0
