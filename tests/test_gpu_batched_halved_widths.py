"""The adaptive width of the persistent batched launch where halving leaves the
multiples of four (12 -> 6, 4 -> 2 -> 1, 20 -> 10, 36 -> 18 -> 9, 60 -> 30):
partial tiles of the Gram matrix, of Z and of Y, in groups whose slots are
added directly and in groups that exchange.

Inputs: all columns but the first b_final are combinations of those plus 1e-12
of noise, so every wider first panel has a Gram matrix singular by nine orders
of magnitude beyond the bound, and from b_final on every panel has a condition
number below 100 (the bound is 1e7): no decision depends on rounding, and the
final width has to be the oracle's.  Tolerances: as for every factorisation.
"""
import numpy as np
import pytest

from _helpers import orth_err, resid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _matrix(m, n, b_final, seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((m, n)) / np.sqrt(m)
    A[:, b_final:] = A[:, :b_final] @ rng.standard_normal((b_final, n - b_final)) + 1e-12 * A[:, b_final:]
    return np.asfortranarray(A)


@pytest.mark.parametrize("group", [0, 4])
@pytest.mark.parametrize("m,n,b,b_final", [(3001, 24, 12, 6), (2000, 8, 4, 2), (1000, 8, 4, 1), (5003, 40, 20, 10),
                                           (4000, 36, 36, 9), (6000, 60, 60, 30), (20000, 120, 60, 30)])
def test_halved_width_is_not_a_multiple_of_four(cuda_lib, oracle, m, n, b, b_final, group):
    P = cuda_lib
    A = _matrix(m, n, b_final, seed=9300 + n)
    _, _, bo = oracle.mcqr2gs_halving(A, b)
    assert bo == b_final
    ws = torch.empty(P.batched_workspace_size([m], [n], [b], halving=True, group=group), dtype=torch.uint8,
                     device="cuda")
    Q, R = P.factor_batched([torch.from_numpy(A).cuda()], [b], workspace=ws, halving=True, group=group)[0]
    assert P.batched_panel_widths(ws, 1) == [b_final]
    Qn, Rn = Q.cpu().numpy(), R.cpu().numpy()
    assert orth_err(Qn) <= 1e-13 and resid(A, Qn, Rn) <= 1e-14
    assert np.all(np.tril(Rn, -1) == 0) and np.all(np.diag(Rn) > 0)
