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
    L.handout_starved.argtypes = [C.c_ulonglong, C.c_ulonglong, C.c_void_p]
    return L


@pytest.mark.parametrize("warps, n_ligs, blocks, units, item_units, slots", [
    (1, 1, 1, 1, 1, 1), (3, 1, 4, 7, 3, 1), (4, 6, 8, 3, 1, 1), (4, 7, 40, 3, 2, 2), (4, 9, 20, 2, 1, 3)])
def test_units_are_handed_out_once_and_lanes_agree(lib, warps, n_ligs, blocks, units, item_units, slots):
    out = np.zeros(5, np.int32)
    lib.handout_job(warps, n_ligs, blocks, units, item_units, slots, out.ctypes.data_as(C.c_void_p))
    once, total, split, wrong, err = out.tolist()
    assert (split, wrong, err) == (0, 0, 0)
    assert once == total == blocks * n_ligs * units


@pytest.mark.parametrize("busy_s, wait_s, by_the_waiting_warp", [(20, 30, 1), (1, 30, 1), (20, 5, 0)])
def test_a_warp_waits_for_a_slot_as_long_as_the_launch_allows(lib, busy_s, wait_s, by_the_waiting_warp):
    """A slot held for 20 s does not cost the CTA the warp that waits for it unless the launch's bound is shorter;
    either way every unit is done."""
    out = np.zeros(3, np.int32)
    lib.handout_starved(busy_s * 10 ** 9, wait_s * 10 ** 9, out.ctypes.data_as(C.c_void_p))
    assert out.tolist() == [by_the_waiting_warp, 2, 0]


def test_step_blocks_are_short_and_few_enough(lib):
    block = lib.handout_step_block
    for steps in (1, 7, 8, 100, 256, 257, 1000, 2000, 16384):       # 1/32 of the steps, at least 8
        assert block(steps, 0, 0, 1000) == max(8, -(-steps // 32))
    for steps in (1, 25, 400, 401, 2000, 8192):                      # a fixed CTA: 1/16, at least 25
        assert block(steps, 1, 0, 1000) == block(steps, 1, 1, 1000) == max(25, -(-steps // 16))
    for steps in (20000, 1000000, 2 ** 31 - 1):                      # never longer than 512 where blocks are handed over
        for items in (1, 64, 40000, 10 ** 6):
            for fixed in (0, 1):
                b = block(steps, fixed, 0, items)
                assert 0 < -(-steps // b) * items < 2 ** 31 - 10 ** 6
                assert b <= 512 or -(-steps // 512) * items > 2 ** 30 - items
        assert block(steps, 0, 1, 64) == steps                       # every chain resident: one block
