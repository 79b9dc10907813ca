"""How launches over items of different sizes are cut into runs (pv_runs.h): every item with blocks is in one run whose
grid covers it, no run has more than twice its items' blocks but for a few, equal items share one launch up to the
grid's limit, and mixed sizes take a launch or two more rather than a grid of the largest for all. Host code."""
import ctypes as C
import os
import random
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2506_20043_gb300", "csrc")
WASTE = 8192


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("runs") / "libruns.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                           os.path.join(ROOT, "tests", "csrc", "launch_runs.cpp"), "-o", out])
    return C.CDLL(out)


def _cut(lib, sizes, first=0, fail_at=-1):
    x = np.array([s[0] for s in sizes], np.int64)
    y = np.array([s[1] for s in sizes], np.int64)
    runs, n = np.zeros((len(sizes) + 1, 4), np.int64), C.c_int()
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)   # noqa: E731
    status = lib.cut_runs(first, len(sizes) - first, ptr(x), ptr(y), fail_at, ptr(runs), len(runs), C.byref(n))
    return status, runs[:n.value].tolist()


def _check(sizes, runs, first=0):
    at = first
    for r0, m, x, y in runs:
        assert all(s[0] * s[1] == 0 for s in sizes[at:r0]) and 1 <= m <= 65535
        items = sizes[r0:r0 + m]
        assert x == max(s[0] for s in items) and y == max(s[1] for s in items)
        work = sum(s[0] * s[1] for s in items)
        assert m == 1 or x * y * m - work <= work + WASTE
        at = r0 + m
    assert all(s[0] * s[1] == 0 for s in sizes[at:])


def test_equal_items_share_a_launch(lib):
    for n in (1, 2, 10, 65535):
        assert _cut(lib, [(337, 6)] * n) == (0, [[0, n, 337, 6]])
    assert [r[1] for r in _cut(lib, [(5, 1)] * 65536)[1]] == [65535, 1]


def test_one_large_item_among_small_ones(lib):
    for at in (0, 50, 100):
        sizes = [(38, 1)] * 100
        sizes.insert(at, (62500, 1))
        status, runs = _cut(lib, sizes)
        _check(sizes, runs)
        assert status == 0 and len(runs) <= 3
        assert sum(m * x * y for _, m, x, y in runs) < 2.1 * sum(s[0] for s in sizes) + WASTE


def test_random_sizes(lib):
    rng = random.Random(5)
    for _ in range(200):
        sizes = [(int(10 ** rng.uniform(-0.5, 5)), rng.choice((0, 1, 1, 8, 2816))) for _ in range(rng.randint(1, 60))]
        first = rng.randint(0, len(sizes) - 1)
        status, runs = _cut(lib, sizes, first)
        assert status == 0
        _check(sizes, runs, first)


def test_a_failed_launch_ends_the_loop(lib):
    sizes = [(10 ** 6, 1), (1, 1), (1, 1), (10 ** 6, 1)]
    assert _cut(lib, sizes)[1] == [[0, 2, 10 ** 6, 1], [2, 2, 10 ** 6, 1]]
    status, runs = _cut(lib, sizes, fail_at=0)
    assert status == 7 and len(runs) == 1
    assert _cut(lib, [(0, 1), (3, 0)])[1] == []
