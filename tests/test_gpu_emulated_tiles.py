"""The emulated products at the edges of their tiles and stages: contractions
on both sides of the four stages that keep X in shared memory (K = 128), a
block's run of column tiles ending inside a row tile, partial row and column
tiles, fixed-point values at the top of their scale, and level sums of the
longest contraction.

Tolerance: R and Q agree with Householder QR to the forward error of the
method, a small multiple of kappa * u with kappa = 1e3: 1e-11 leaves two
orders of magnitude.  One column: its Gram entry is a sum of m equal squares
x^2 >= 2^-2 of the scale, off by at most the neglected digit products (10 x 256
x 32^9 of 2^108) and the representation, 2^-49.6 of it; the root halves that,
and the few roundings of the second pass and the solve add less than 2^-51.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _matrix(m, n, kappa, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    G = torch.randn((n, m), generator=gen, dtype=torch.float64, device="cuda").t()
    V = torch.linalg.qr(torch.randn((n, n), generator=gen, dtype=torch.float64, device="cuda")).Q
    s = torch.logspace(0, -torch.log10(torch.tensor(kappa)).item(), n, dtype=torch.float64, device="cuda") / m ** 0.5
    return (V @ (s[:, None] * G.t())).t()


@pytest.mark.parametrize("m,n,b", [
    (129, 96, 32), (4095, 66, 33), (4097, 512, 128), (20001, 516, 129), (30011, 387, 129), (40000, 310, 31),
    (5000, 1280, 160), (100003, 192, 64), (152 * 128 * 3 + 77, 288, 96)])
def test_emulated_matches_householder(cuda_lib, m, n, b):
    A = _matrix(m, n, 1e3, m + n)
    Q, R = cuda_lib.factor(A, b, emulated=True)
    Qh, Rh = torch.linalg.qr(A)
    d = torch.where(torch.diagonal(Rh) < 0, -1.0, 1.0).to(torch.float64)
    assert (torch.linalg.norm(R - d[:, None] * Rh) / torch.linalg.norm(Rh)).item() < 1e-11
    assert (Q - Qh * d).abs().max().item() < 1e-11


@pytest.mark.parametrize("value", [1.0, 1.0 - 2.0 ** -53, 1.0 + 2.0 ** -52, 1.9375, 15.5 / 16, -(1.0 - 2.0 ** -20)])
@pytest.mark.parametrize("m", [4096, 12345])
def test_emulated_top_of_scale(cuda_lib, value, m):
    """One column of equal entries: R = |value| sqrt(m), every level sum at its largest."""
    A = torch.full((1, m), value, dtype=torch.float64, device="cuda").t()
    Q, R = cuda_lib.factor(A, 1, emulated=True)
    want = abs(value) * m ** 0.5
    assert abs(R.item() - want) <= want * 2.0 ** -50
    assert (Q * R.item() - A).abs().max().item() <= abs(value) * 2.0 ** -50
