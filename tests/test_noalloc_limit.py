"""Which sizes cqr_factor_noalloc takes: every factorisation whose
cqr_workspace_size() is at most CQR_NOALLOC_SCRATCH_BYTES, as its declaration
says (and, for short matrices, up to 16 MiB more)."""
import ctypes

import pytest

import paper_2405_04237_gb300 as P
from paper_2405_04237_gb300 import _capi

torch = pytest.importorskip("torch")


@pytest.mark.skipif(torch.cuda.is_available(), reason="made-up addresses: for machines that cannot launch")
def test_every_fitting_size_is_taken():
    """Without a GPU a call that is not refused ends at the lookup of the array."""
    L = P.load()
    vp = ctypes.c_void_p
    A, Q, R = 1 << 40, 1 << 41, 1 << 42
    refused = 0
    for variant in ("mcqr2gs", "cqr2gs"):
        for m in (2000, 20000, 100000, 1 << 20):
            for b in (8, 12, 24, 36, 40, 48, 72, 90, 128):
                for k in range(1, 60):
                    n = k * b
                    if n > m:
                        break
                    need = P.workspace_size(m, n, b, variant)
                    rc = L.cqr_factor_noalloc(m, n, vp(A), m, b, vp(Q), m, vp(R), n, P.VARIANTS[variant], None, None)
                    refused += rc == _capi.ERR_NOALLOC_TOO_LARGE
                    if need <= _capi.NOALLOC_SCRATCH_BYTES:
                        assert rc != _capi.ERR_NOALLOC_TOO_LARGE, (variant, m, n, b, need)
                    elif need > _capi.NOALLOC_SCRATCH_BYTES + (16 << 20):
                        assert rc == _capi.ERR_NOALLOC_TOO_LARGE, (variant, m, n, b, need)
    assert refused > 0


@pytest.mark.gpu
def test_fitting_size_runs(cuda_lib):
    """A width whose tiles, cut to the product, need less than the fixed tiles of 64 would."""
    m, n, b = 50000, 1800, 36
    assert P.workspace_size(m, n, b, "cqr2gs") <= _capi.NOALLOC_SCRATCH_BYTES
    A = P.colmajor(torch.randn((m, n), dtype=torch.float64, device="cuda"))
    Q, R = P.empty_colmajor(m, n, "cuda"), P.empty_colmajor(n, n, "cuda")
    status = torch.full((1,), -7, dtype=torch.int32, device="cuda")
    rc = P.load().cqr_factor_noalloc(m, n, P._ptr(A), m, b, P._ptr(Q), m, P._ptr(R), n, P.VARIANTS["cqr2gs"],
                                     P._ptr(status), P._stream())
    assert rc == 0
    Qw, Rw = P.factor(A, b, "cqr2gs")
    assert int(status.item()) == 0 and torch.equal(Q, Qw) and torch.equal(R, Rw)
