"""The product kernel's micro-tiles (2 x 2, single entries) on both sides of the
line between them, through factorisations whose updates and R products
fall there, and the same calls captured into a CUDA graph: the launches that
start before the one ahead of them has ended give the eager result bit for bit.

Tolerance: as in the parity tests, the forward error at kappa = 1e3.
"""
import pytest

from _helpers import rel_diff
from testmatrices import make_test_matrix

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,b,kw", [
    (513, 6, 3, {}), (2000, 16, 4, {}), (4864, 32, 16, {}), (9729, 24, 8, {}), (20000, 64, 16, {"lookahead": True}),
    (19456, 128, 64, {}), (3000, 256, 128, {}), (5001, 60, 12, {"variant": "cqr2gs"}), (2500, 130, 0, {"variant": "scqr3"}),
    (9000, 96, 48, {"emulated": True})])
def test_products_and_capture(cuda_lib, oracle, m, n, b, kw):
    P = cuda_lib
    A = make_test_matrix(m, n, 1e3, seed=8300 + n)
    At = P.colmajor(torch.from_numpy(A).cuda())
    Q, R = P.factor(At, b, **kw)
    variant = kw.get("variant", "mcqr2gs")
    if variant == "scqr3":
        Qo, Ro = oracle.scqr3(A)
    else:
        Qo, Ro = getattr(oracle, variant)(A, b)
    assert rel_diff(R.cpu().numpy(), Ro) < 1e-11 and abs(Q.cpu().numpy() - Qo).max() < 1e-11
    size = {k: v for k, v in kw.items() if k != "lookahead"}
    out = (P.empty_colmajor(m, n, "cuda"), P.empty_colmajor(n, n, "cuda"))
    ws = torch.empty(P.workspace_size(m, n, b, **size), dtype=torch.uint8, device="cuda")
    P.factor(At, b, out=out, workspace=ws, check=False, **kw)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        P.factor(At, b, out=out, workspace=ws, check=False, **kw)
    out[0].zero_()
    out[1].zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out[0], Q) and torch.equal(out[1], R)
