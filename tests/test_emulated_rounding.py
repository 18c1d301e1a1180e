"""The one rounding of an emulated product (group_value): the exact integer sum
g0 + 2^30 g1 of its level groups, |g0| < 2^51 and |g1| < 2^46, times a power of
two, to the nearest double, halves to even -- against Python's integers."""
import ctypes
import math
import os
import random
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2405_04237_gb300", "csrc")
SCALE = -108 + 45  # of the sum, beside the two operands' exponents


@pytest.fixture(scope="module")
def group_value(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("group_value") / "group_value.so")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC",
                           "-I" + os.path.join(HERE, "device_on_cpu"), "-I" + CSRC,
                           os.path.join(HERE, "device_on_cpu", "group_value.cpp"), "-o", so])
    lib = ctypes.CDLL(so)

    def call(pairs, exy):
        n = len(pairs)
        out = (ctypes.c_double * n)()
        lib.group_values(n, (ctypes.c_longlong * n)(*[a for a, _ in pairs]),
                         (ctypes.c_longlong * n)(*[b for _, b in pairs]), (ctypes.c_int * n)(*[exy] * n), out)
        return list(out)

    return call


def _check(group_value, pairs, exy):
    for (g0, g1), got in zip(pairs, group_value(pairs, exy)):
        want = math.ldexp(float(g0 + (g1 << 30)), exy + SCALE)  # float(int) rounds half to even
        assert got == want, (g0, g1, exy, got, want)


@pytest.mark.parametrize("exy", [0, 63, -700, 900])
def test_random_sums(group_value, exy):
    rng = random.Random(5)
    pairs = []
    for _ in range(20000):
        a, b = rng.randint(1, 51), rng.randint(0, 46)
        pairs.append((rng.randint(-(2 ** a) + 1, 2 ** a - 1), rng.randint(-(2 ** b), 2 ** b)))
    _check(group_value, pairs, exy)


def test_ties_and_their_neighbours(group_value):
    """54 significant bits ending in 1, at every position of the 76 bits, and one unit to either side."""
    rng = random.Random(6)
    pairs = []
    for shift in range(0, 22):
        for _ in range(400):
            tie = (rng.getrandbits(53) | 1 << 52) * 2 + 1
            for d in (-1, 0, 1):
                total = rng.choice((-1, 1)) * ((tie << shift) + (d if shift else 0))
                g0 = total % (1 << 30) - rng.choice((0, 1 << 30))
                pairs.append((g0, (total - g0) >> 30))
    assert all(abs(a) < 2 ** 51 and abs(b) <= 2 ** 46 for a, b in pairs)
    _check(group_value, pairs, 10)
