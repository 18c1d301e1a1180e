"""The persistent batched launch's default schedule (groups of several sizes:
nodes of a tree over the CTAs) at its edges: one matrix alone (all CTAs, fewer
rows than CTAs too), one large matrix among many small ones, more matrices
than CTAs, every panel width class, and the in-CTA sums' thread splits.

Tolerance: Q and R agree with the oracle to the forward error of the method, a
small multiple of kappa * u with kappa = 1e3: 1e-11 leaves two orders of
magnitude.
"""
import numpy as np
import pytest

from _helpers import rel_diff
from testmatrices import make_test_matrix

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = {
    "one": [(70001, 128, 64)],
    "one_short": [(130, 128, 128)],
    "fewer_rows_than_ctas": [(100, 16, 4), (64, 64, 64)],
    "large_and_small": [(60000, 128, 32)] + [(300 + 37 * i, 16 + 4 * (i % 5), 4) for i in range(12)],
    "many": [(200 + 13 * i, (16, 20, 32, 64)[i % 4], 4) for i in range(180)],
    "widths": [(3000 + 101 * i, n, b) for i, (n, b) in enumerate(
        [(4, 4), (8, 4), (12, 12), (36, 12), (40, 20), (64, 16), (96, 48), (100, 100), (124, 4), (128, 8)])],
}


@pytest.mark.parametrize("name", sorted(SHAPES))
def test_default_schedule_matches_the_oracle(cuda_lib, oracle, name):
    shapes = SHAPES[name]
    As = [make_test_matrix(m, n, 1e3, seed=8100 + i) for i, (m, n, b) in enumerate(shapes)]
    Ts = [torch.from_numpy(np.asfortranarray(A)).cuda() for A in As]
    res = cuda_lib.factor_batched(Ts, [b for _, _, b in shapes])
    again = cuda_lib.factor_batched(Ts, [b for _, _, b in shapes])
    for A, (Q, R), (Q2, R2), (m, n, b) in zip(As, res, again, shapes):
        assert torch.equal(Q, Q2) and torch.equal(R, R2)
        Qo, Ro = oracle.mcqr2gs(A, b)
        Rn = R.cpu().numpy()
        assert np.all(np.tril(Rn, -1) == 0)
        assert rel_diff(Rn, Ro) < 1e-11 and np.abs(Q.cpu().numpy() - Qo).max() < 1e-11, (m, n, b)


def test_default_schedule_statuses(cuda_lib):
    """A breakdown in one matrix leaves the others of its group alone."""
    As = [make_test_matrix(2000, 32, 1e2, seed=8200 + i) for i in range(170)]
    As[3][:, 9] = 0.0
    As[160][:, 30] = 0.0
    status = torch.zeros(170, dtype=torch.int32, device="cuda")
    cuda_lib.factor_batched([torch.from_numpy(np.asfortranarray(A)).cuda() for A in As], 8, check=False, status=status)
    want = [0] * 170
    want[3], want[160] = 10, 31
    assert status.tolist() == want
