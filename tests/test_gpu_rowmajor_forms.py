"""Row-major tensors that are no plain matrix in memory take torch's own copy,
as before the library copied row-major matrices itself: zeros without storage
and tensors of function transforms (refused by torch)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _problem(P, m=500, n=12):
    gen = torch.Generator(device="cuda").manual_seed(9600)
    A = torch.randn((m, n), generator=gen, dtype=torch.float64, device="cuda")
    dR = torch.randn((n, n), generator=gen, dtype=torch.float64, device="cuda").triu()
    return A, dR


def test_zeros_without_storage(cuda_lib):
    P = cuda_lib
    A, dR = _problem(P)
    Q, R = P.factor(A, 4)
    zero = torch._efficientzerotensor(A.shape, dtype=torch.float64, device="cuda")
    assert torch.equal(P.backward(Q, R, zero, dR), P.backward(Q, R, torch.zeros_like(A), dR))


def test_transform_is_refused_by_torch(cuda_lib):
    P = cuda_lib
    A, _ = _problem(P)
    with pytest.raises(RuntimeError):
        torch.func.vmap(lambda x: P.factor(x, 4)[1])(torch.stack([A, A]))


def test_no_private_name_is_needed(cuda_lib, monkeypatch):
    P = cuda_lib
    A, _ = _problem(P)
    want = P.factor(A, 4)
    monkeypatch.delattr(torch._C._functorch, "is_functorch_wrapped_tensor")
    got = P.factor(A, 4)
    assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1])
