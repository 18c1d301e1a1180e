"""The one-block Cholesky elimination (chol_trapezoid, shared by every path) as
compiled for the CPU, with the warps of the block in chosen orders between two
barriers: the first warp ahead of all others, behind them, and shuffled.  No
order may change a bit of the result: a step in which one warp reads what
another writes would.

Tolerance of the values: the elimination and the reference (the row-by-row
definition in long double) differ by the rounding of at most kb terms per
entry, amplified by the condition number of W = I + G^T G / (4 n), below 3:
1e-13 leaves a factor of ten at kb = 128.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2405_04237_gb300", "csrc")


@pytest.fixture(scope="module")
def trapezoid(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("trapezoid") / "trapezoid.so")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-Wno-unknown-pragmas", "-shared", "-fPIC",
                           "-I" + os.path.join(HERE, "device_on_cpu"), "-I" + CSRC,
                           os.path.join(HERE, "device_on_cpu", "trapezoid.cpp"), "-o", so])
    lib = ctypes.CDLL(so)
    lib.trapezoid.argtypes = [ctypes.c_int] + [ctypes.c_void_p] + 2 * [ctypes.c_int] + 2 * [ctypes.c_void_p]

    def call(T, order, W, nx):
        kb = W.shape[0]
        F, dg, o = W.copy(), np.zeros(kb), np.ascontiguousarray(order, dtype=np.int32)
        r = lib.trapezoid(T, o.ctypes.data, kb, nx, F.ctypes.data, dg.ctypes.data)
        F[np.arange(kb), np.arange(kb)] = dg
        return r, np.triu(F)

    return call


def _gram(kb, nx, seed):
    n = kb + nx
    G = np.random.default_rng(seed).standard_normal((4 * n, n))
    return np.ascontiguousarray((np.eye(n) + G.T @ G / (4.0 * n))[:kb])


def _factor_rows(W):
    kb, n = W.shape
    U = np.zeros((kb, n), dtype=np.longdouble)
    for j in range(kb):
        row = W[j].astype(np.longdouble) - U[:j, j] @ U[:j]
        U[j, j:] = row[j:] / np.sqrt(row[j])
    return U


def _orders(T):
    w = T // 32
    rng = np.random.default_rng(T)
    return [np.arange(w), np.arange(w)[::-1]] + [rng.permutation(w) for _ in range(2)]


# one block (256 threads, up to 64 columns), a tile of the cluster with its share of further columns, the batched
# launch (512 threads, up to 128 columns); one to five warps hold the pivot rows
@pytest.mark.parametrize("T,kb,nx", [(256, 1, 0), (256, 2, 0), (256, 32, 0), (256, 33, 0), (256, 35, 0), (256, 64, 0),
                                     (256, 32, 1), (256, 32, 60), (256, 7, 40), (512, 36, 0), (512, 100, 0),
                                     (512, 128, 0)])
def test_any_warp_order_gives_the_factor(trapezoid, T, kb, nx):
    W = _gram(kb, nx, seed=100 * kb + nx)
    want = _factor_rows(W)
    first = None
    for order in _orders(T):
        r, U = trapezoid(T, order, W, nx)
        assert r == -1
        assert np.abs(U - want).max() < 1e-13, order
        first = U if first is None else first
        assert np.array_equal(U, first), order


@pytest.mark.parametrize("T,kb,nx,row", [(256, 64, 0, 8), (256, 64, 0, 9), (256, 32, 60, 31), (512, 128, 0, 40)])
def test_breakdown_in_any_warp_order(trapezoid, T, kb, nx, row):
    W = _gram(kb, nx, seed=17)
    W[row, row] = -1.0
    want = _factor_rows(W[:row])
    for order in _orders(T):
        r, U = trapezoid(T, order, W, nx)
        assert r == row
        assert np.abs(U[:row] - want).max() < 1e-13, order


# The whole range of pivots: down to subnormal Gram entries (columns of norm 1e-158), up to the largest.  W keeps
# log2(s) + 1074 bits there and every term of the elimination is rounded to 2^-1074: kb of them move an entry of U by
# a multiple (the condition number, below 3, and a factor for the root) of kb 2^-1074 / s of its scale sqrt(s).
@pytest.mark.parametrize("T,kb,nx", [(256, 16, 0), (256, 40, 0), (256, 32, 20), (512, 64, 0)])
@pytest.mark.parametrize("e", [-1050, -1040, -1026, -1023, -1022, -600, 0, 600, 1020, 1021])
def test_pivots_of_any_size(trapezoid, T, kb, nx, e):
    s = np.ldexp(1.0, e)
    W = _gram(kb, nx, seed=29) * s
    scale = np.sqrt(np.longdouble(2.0) ** e)
    want = _factor_rows(np.ldexp(W, -e)) * scale  # exact: a power of two
    r, U = trapezoid(T, np.arange(T // 32), W, nx)
    assert r == -1
    assert np.abs(U - want).max() <= 8 * kb * (2.0 ** (-1074 - e) + 2.0 ** -53) * scale
