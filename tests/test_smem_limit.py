"""The per-kernel shared-memory limits that launches raise (pv_smem.h), from several threads at once: none lowers
the limit behind another, so no launch finds less than it asked for. Host code, no GPU."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2506_20043_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("smem") / "libsmem.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-pthread", "-I", CSRC,
                           os.path.join(ROOT, "tests", "csrc", "smem_limit.cpp"), "-o", out])
    return C.CDLL(out)


@pytest.mark.parametrize("threads", [2, 3, 8])
def test_no_thread_lowers_the_limit_of_another(lib, threads):
    assert lib.refused_launches(threads, 400) == 0


def test_a_failed_raise_is_reported_and_tried_again(lib):
    assert lib.failed_raise() == 73
