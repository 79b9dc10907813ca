"""How the warps of a CTA of the batched search take their chains (pv_handout.cuh), run on the host with every lane
of every warp a thread of its own (tests/csrc/handout.cpp): each unit is handed out once, the lanes of a warp always
agree on what they took although other warps give ligand slots back meanwhile, and no slot is restaged while a
warp works on it."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2506_20043_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("handout") / "libhandout.so")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-pthread", "-w", "-I", CSRC, "-I", cuda_inc,
                           os.path.join(ROOT, "tests", "csrc", "handout.cpp"), "-ldl", "-o", out])
    L = C.CDLL(out)
    return L


@pytest.mark.parametrize("warps, n_ligs, blocks, units, item_units, slots", [
    (1, 1, 1, 1, 1, 1), (3, 1, 4, 7, 3, 1), (4, 6, 8, 3, 1, 1), (4, 7, 40, 3, 2, 2), (4, 9, 20, 2, 1, 3)])
def test_units_are_handed_out_once_and_lanes_agree(lib, warps, n_ligs, blocks, units, item_units, slots):
    out = np.zeros(5, np.int32)
    lib.handout_job(warps, n_ligs, blocks, units, item_units, slots, out.ctypes.data_as(C.c_void_p))
    once, total, split, wrong, err = out.tolist()
    assert (split, wrong, err) == (0, 0, 0)
    assert once == total == blocks * n_ligs * units
