"""The runtime choice of the second CholeskyQR pass, its decision itself: the
word at byte 256 of the workspace, set by the last panel's Cholesky kernel, for
panels of one block (up to 64 columns) and of the cluster of eight (above).

Orthogonal columns with power-of-two norms: every step is exact, the second
Gram matrix is I, the solve is skipped and R = diag(norms) bit for bit.
kappa = 1e5: the second factor is 1e-6 away from I (kappa^2 u), far outside 8u:
nothing is skipped and the results are the default schedule's bit for bit.
"""
import numpy as np
import pytest

from _helpers import hadamard
from testmatrices import make_test_matrix

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WIDTHS = [(16, 16), (64, 64), (65, 65), (100, 100), (300, 300), (200, 100), (128, 64)]


def _adaptive(P, A, b):
    m, n = A.shape
    T = torch.from_numpy(np.asfortranarray(A)).cuda()
    ws = torch.empty(P.workspace_size(m, n, b), dtype=torch.uint8, device="cuda")
    Q, R = P.factor(T, b, workspace=ws, adaptive=True)
    return T, Q, R, int(ws[256:260].view(torch.int32).item())


@pytest.mark.parametrize("n,b", WIDTHS)
def test_identity_is_skipped(cuda_lib, n, b):
    rng = np.random.default_rng(9400 + n)
    m = 4096
    Q0 = hadamard(m)[:, np.sort(rng.choice(m, size=n, replace=False))] / 64.0
    d = 2.0 ** rng.integers(-3, 4, size=n)
    _, Q, R, skipped = _adaptive(cuda_lib, Q0 * d, b)
    assert skipped == 1
    assert np.array_equal(R.cpu().numpy(), np.diag(d)) and np.array_equal(Q.cpu().numpy(), Q0)


@pytest.mark.parametrize("n,b", WIDTHS)
def test_distant_factor_is_not_skipped(cuda_lib, n, b):
    P = cuda_lib
    T, Q, R, skipped = _adaptive(P, make_test_matrix(4000, n, 1e5, seed=9500 + n), b)
    assert skipped == 0
    Qd, Rd = P.factor(T, b)
    assert torch.equal(Q, Qd) and torch.equal(R, Rd)
