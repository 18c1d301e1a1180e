"""Matrices whose Gram matrices fall among the subnormal numbers, or near the
top of the range: scaled by a power of two, A = Q R only changes R's scale.

Tolerances: the first Cholesky factor of 2^-516 A carries 40 bits, and the
second CholeskyQR takes the panel back to working precision: ||I - Q^T Q|| <=
1e-13 and residual <= 1e-14 as for any matrix, R to kappa (10) times these.
"""
import numpy as np
import pytest

from _helpers import orth_err, rel_diff, resid
from testmatrices import make_test_matrix

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("m,n,b", [(2000, 16, 16), (3001, 40, 40), (4000, 96, 96), (5000, 128, 32)])
@pytest.mark.parametrize("e", [-516, 510])
def test_scaled_matrix(cuda_lib, oracle, m, n, b, e, batched):
    P = cuda_lib
    A = make_test_matrix(m, n, 10.0, seed=9100 + n)
    T = torch.from_numpy(np.asfortranarray(np.ldexp(A, e))).cuda()
    Q, R = P.factor_batched([T], [b])[0] if batched else P.factor(T, b)
    Qn, Rn = Q.cpu().numpy(), np.ldexp(R.cpu().numpy(), -e)
    _, Ro = oracle.mcqr2gs(A, b)
    assert orth_err(Qn) <= 1e-13 and resid(A, Qn, Rn) <= 1e-14
    assert rel_diff(Rn, Ro) <= 1e-12
