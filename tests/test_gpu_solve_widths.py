"""The triangular solves at every register width (panel widths rounded up to
multiples of four, up to the 64 columns of a block) and at the edges of a block
of 128 rows, forward through a factorisation and transposed through the adjoint.

Tolerance: as in the parity tests, the forward error at kappa = 1e3 (1e-11 for Q
and R; 1e-10 relative for the adjoint, whose solve multiplies it by kappa(R)
times u once more)."""
import numpy as np
import pytest

from _helpers import rel_diff
from testmatrices import make_test_matrix

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,b", [(127, 1), (128, 3), (129, 4), (255, 5), (257, 12), (1000, 17), (384, 28), (385, 31),
                                 (900, 36), (1025, 41), (1151, 44), (1153, 47), (2000, 52), (640, 57), (641, 60), (1281, 63),
                                 (1280, 64), (3000, 65), (2500, 124)])
def test_solves_match_the_oracle(cuda_lib, oracle, m, b):
    A = make_test_matrix(m, b, 1e3, seed=8400 + b)
    Q, R = cuda_lib.factor(torch.from_numpy(A).cuda(), b)
    Qo, Ro = oracle.mcqr2gs(A, b)
    assert rel_diff(R.cpu().numpy(), Ro) < 1e-11 and np.abs(Q.cpu().numpy() - Qo).max() < 1e-11
    rng = np.random.default_rng(b)
    dQ, dR = rng.standard_normal((m, b)), np.triu(rng.standard_normal((b, b)))
    dA = cuda_lib.backward(Q, R, torch.from_numpy(dQ).cuda(), torch.from_numpy(dR).cuda()).cpu().numpy()
    assert rel_diff(dA, oracle.backward(Q.cpu().numpy(), R.cpu().numpy(), dQ, dR)) < 1e-10
