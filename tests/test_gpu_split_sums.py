"""The split-m products at the edges of their plans: widths on both sides of
each thread mapping of the Gram kernel (every tile a main tile, or main and
extra tiles; 128 or 512 threads), row counts from one short block per SM to
several staged blocks each, and projection tiles of every padding.

Tolerance: R and Q agree with the oracle to the forward error of the method,
a small multiple of kappa * u with kappa = 1e3, so 1e-11 leaves two orders
of magnitude.
"""
import numpy as np
import pytest

from _helpers import rel_diff
from testmatrices import make_test_matrix

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,b", [
    (33, 13, 13), (64, 64, 4), (1000, 9, 1), (2001, 16, 4), (4999, 51, 17), (3001, 60, 30), (5003, 66, 33),
    (7001, 96, 48), (8823, 64, 64), (8825, 130, 65), (4700, 176, 88), (4801, 178, 89), (33500, 64, 32),
    (120100, 32, 16), (20011, 75, 15)])
def test_split_sums_match_the_oracle(cuda_lib, oracle, m, n, b):
    A = make_test_matrix(m, n, 1e3, seed=7000 + n)
    Q, R = cuda_lib.factor(torch.from_numpy(A).cuda(), b)
    Qo, Ro = oracle.mcqr2gs(A, b)
    Rn = R.cpu().numpy()
    assert np.all(np.tril(Rn, -1) == 0)
    assert rel_diff(Rn, Ro) < 1e-11 and np.abs(Q.cpu().numpy() - Qo).max() < 1e-11
