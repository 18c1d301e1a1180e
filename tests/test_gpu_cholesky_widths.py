"""The Cholesky kernels at the edges of their panel widths: one block up to 64
columns (with one or two pivot warps), a cluster of eight above (row tiles of
32, ragged last tiles, up to 512), exact square roots and quotients, a
breakdown inside the last tile, and the identity rule of the runtime
repetition choice for a wide panel.

Tolerances: 1e-11 element-wise at kappa = 1e3 (forward error a small multiple
of kappa * u); exact inputs bit for bit.
"""
import numpy as np
import pytest

from _helpers import exact_qr_case, rel_diff
from testmatrices import make_test_matrix

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _t(A):
    return torch.from_numpy(np.asfortranarray(A)).cuda()


@pytest.mark.parametrize("b", [1, 2, 32, 33, 34, 63, 64, 65, 95, 96, 97, 129, 250, 511, 512])
def test_widths_match_the_oracle(cuda_lib, oracle, b):
    A = make_test_matrix(1537, b, 1e3, seed=7300 + b)
    Q, R = cuda_lib.factor(_t(A), b)
    Qo, Ro = oracle.mcqr2gs(A, b)
    assert rel_diff(R.cpu().numpy(), Ro) < 1e-11 and np.abs(Q.cpu().numpy() - Qo).max() < 1e-11


@pytest.mark.parametrize("m,n", [(1024, 64), (4096, 160), (4096, 512)])
def test_exact_wide_panels_bitwise(cuda_lib, m, n):
    A, Q0, R0 = exact_qr_case(m, n, seed=m + n)
    Q, R = cuda_lib.factor(_t(A), n)
    if n <= 64:  # wider: the exact factor's entries outgrow 53 bits in the Gram matrix
        assert np.array_equal(R.cpu().numpy(), R0) and np.array_equal(Q.cpu().numpy(), Q0)
    else:
        assert rel_diff(R.cpu().numpy(), R0) < 1e-9


@pytest.mark.parametrize("b,col", [(64, 63), (96, 40), (250, 249), (512, 300)])
def test_breakdown_column(cuda_lib, oracle, b, col):
    A = make_test_matrix(2000, b, 1e2, seed=7400 + b)
    A[:, col] = 0.0
    with pytest.raises(cuda_lib.CQRError) as e:
        cuda_lib.factor(_t(A), b)
    assert e.value.code == col + 1


def test_identity_rule_wide_panel(cuda_lib):
    """Orthonormal columns: the second pass finds U within 8u of I and skips
    its solve; the results equal the default schedule's to rounding."""
    A, _ = np.linalg.qr(np.random.default_rng(7500).standard_normal((4000, 200)))
    Q, R = cuda_lib.factor(_t(A), 100)
    Qa, Ra = cuda_lib.factor(_t(A), 100, adaptive=True)
    assert torch.dist(Q, Qa) < 1e-13 and torch.dist(R, Ra) < 1e-13
