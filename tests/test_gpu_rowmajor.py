"""Row-major inputs: the layout copy (cqr_colmajor) at the edges of its 64 x 32
tiles, bit for bit, and the entry points that take it against the same call on
the column-major matrix."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,pad", [(1, 1, 0), (2, 33, 0), (63, 31, 1), (64, 32, 0), (65, 33, 5), (4097, 1, 0),
                                     (1000, 130, 3), (130, 130, 0)])
def test_copy_is_exact(cuda_lib, m, n, pad):
    P = cuda_lib
    A = torch.randn((m, n + pad), dtype=torch.float64, device="cuda")[:, :n]
    guard = torch.full((n, m + 2), 7.0, dtype=torch.float64, device="cuda")
    Q = guard.t()[:m]  # column-major, ldq = m + 2
    L = P.load()
    assert L.cqr_colmajor(m, n, P._ptr(A), n + pad, P._ptr(Q), m + 2, P._stream()) == 0
    assert torch.equal(Q, A) and bool((guard.t()[m:] == 7.0).all())
    assert L.cqr_colmajor(m, n, P._ptr(A), n - 1, P._ptr(Q), m + 2, P._stream()) == -4
    assert L.cqr_colmajor(m, n, P._ptr(A), n + pad, P._ptr(A), m + 2, P._stream()) == -5


@pytest.mark.parametrize("m,n,b", [(2000, 16, 0), (777, 45, 15), (5000, 128, 32)])
def test_factor_and_backward_equal_column_major(cuda_lib, m, n, b):
    P = cuda_lib
    A = torch.randn((m, n), dtype=torch.float64, device="cuda")
    keep = A.clone()
    Q, R = P.factor(A, b)
    Qc, Rc = P.factor(P.colmajor(A), b)
    assert torch.equal(Q, Qc) and torch.equal(R, Rc) and torch.equal(A, keep)
    wide = torch.randn((m, n + 3), dtype=torch.float64, device="cuda")
    wide[:, :n] = A
    assert torch.equal(P.factor(wide[:, :n], b)[0], Qc)
    dQ, dR = torch.randn_like(A), torch.randn((n, n), dtype=torch.float64, device="cuda").triu()
    assert torch.equal(P.backward(Q, R, dQ, dR), P.backward(Q, R, P.colmajor(dQ), P.colmajor(dR)))
    out = (P.empty_colmajor(m, n, "cuda"), P.empty_colmajor(n, n, "cuda"))
    assert torch.equal(P.factor(A, b, out=out)[0], Qc)
