"""The persistent batched launch's default schedule: the tree of groups or equal
groups of 8, whichever is estimated to be faster, every matrix placed once."""
import ctypes
import os
import random
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2405_04237_gb300", "csrc")


@pytest.fixture(scope="module")
def schedule(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("schedule") / "schedule.so")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I" + CSRC,
                           os.path.join(HERE, "device_on_cpu", "schedule.cpp"), "-o", so])
    lib = ctypes.CDLL(so)

    def call(shapes, grid=152):
        k = len(shapes)
        cnt, placed, seconds = (ctypes.c_int * 16)(), (ctypes.c_int * k)(), (ctypes.c_double * 3)()
        levels = lib.schedule(k, (ctypes.c_int64 * k)(*[s[0] for s in shapes]),
                              (ctypes.c_int64 * k)(*[s[1] for s in shapes]),
                              (ctypes.c_int * k)(*[s[2] for s in shapes]), grid, cnt, placed, seconds)
        assert list(placed) == [1] * k
        return list(cnt)[:levels], list(seconds)

    return call


# measured faster on groups of 8 by 6 % and more (count a multiple of 19), or on the tree
@pytest.mark.parametrize("m,n,b", [(20000, 128, 32), (20000, 128, 64), (100000, 64, 32)])
@pytest.mark.parametrize("count,equal", [(19, True), (38, True), (57, True), (76, True), (1, False), (16, False),
                                         (20, False), (32, False), (40, False), (64, False)])
def test_equal_matrices(schedule, m, n, b, count, equal):
    cnt, _ = schedule([(m, n, b)] * count)
    assert (cnt == [19]) == equal


@pytest.mark.parametrize("grid", [152, 148, 132, 7, 1])
def test_shorter_estimate_is_taken(schedule, grid):
    rng = random.Random(grid)
    for count in (1, 2, 7, 19, 33, 150, 400):
        shapes = [(rng.randint(130, 200000), n, max(4, n // rng.choice((1, 2, 4)))) for n in
                  (rng.choice((16, 32, 64, 128)) for _ in range(count))]
        _, seconds = schedule(shapes, grid)
        assert seconds[0] == min(seconds[1:])
