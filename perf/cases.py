"""The work that a user of this library has it do, as cases that can be timed and compared.

Every case goes through the public entry points of the package.  Matrices are A = G diag(sigma) V^T / sqrt(m) with
G Gaussian, V orthogonal and sigma log-spaced from 1 to 1/kappa, the shape of the library's own test matrices.
kappa stays at or below 1e5, where Q and R are determined to about 1e-11 and two roundings of the same method can
be compared element by element; up to 1e15 only their norms can.
"""
import math

import numpy as np
import torch

import paper_2405_04237_gb300 as cqr


# ------------------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # One small matrix straight from torch (row-major), all defaults, status checked: the smallest call, where
        # launches and the host path count.
        {"name": "factor_2000x16", "kind": "factor", "m": 2000, "n": 16, "b": 0, "variant": "mcqr2gs", "kappa": 1e3,
         "rowmajor": True, "keep": False},
        # The single-matrix workload m = 20,000, n = 64, b = 16 in a loop that keeps its buffers and does not wait.
        {"name": "factor_20000x64", "kind": "factor", "m": 20000, "n": 64, "b": 16, "variant": "mcqr2gs", "kappa": 1e5,
         "rowmajor": False, "keep": True},
        # An ordinary matrix with ragged sizes and the paper's other method.
        {"name": "cqr2gs_30011x90", "kind": "factor", "m": 30011, "n": 90, "b": 15, "variant": "cqr2gs", "kappa": 1e4,
         "rowmajor": True, "keep": False},
        # The call of the README: a tall matrix, row-major input.
        {"name": "factor_1048576x256", "kind": "factor", "m": 1 << 20, "n": 256, "b": 64, "variant": "mcqr2gs",
         "kappa": 1e5, "rowmajor": True, "keep": False},
        # The benchmark's width and panel at the row count of the committed profiles: the largest factorisation.
        {"name": "factor_262144x1024", "kind": "factor", "m": 1 << 18, "n": 1024, "b": 128, "variant": "mcqr2gs",
         "kappa": 1e5, "rowmajor": False, "keep": True},
        # Shifted CholeskyQR3 of a whole matrix: one wide panel, three passes.
        {"name": "scqr3_100000x256", "kind": "factor", "m": 100000, "n": 256, "b": 0, "variant": "scqr3", "kappa": 1e5,
         "rowmajor": False, "keep": True},
        # The tensor-core variant at the benchmark's width, and at a ragged medium size.
        {"name": "emulated_262144x1024", "kind": "emulated", "m": 1 << 18, "n": 1024, "b": 128, "kappa": 1e5,
         "rowmajor": False, "keep": True},
        {"name": "emulated_60013x360", "kind": "emulated", "m": 60013, "n": 360, "b": 72, "kappa": 1e4,
         "rowmajor": False, "keep": True},
        # A batch of uneven matrices, one call, adaptive width: the sizes of the batched workload.
        {"name": "batched_uneven", "kind": "batched", "count": 32, "m_lo": 2000, "m_hi": 200000, "n_step": 0,
         "shapes": 1, "k0": 2, "halving": True},
        # A small batch captured once and replayed, the way a latency-bound program calls it.
        {"name": "graph_small", "kind": "graph", "count": 32, "m_lo": 200, "m_hi": 8000, "n_step": 0, "shapes": 2,
         "k0": 2, "halving": False},
        # A training step through autograd at the differentiable workload's size.
        {"name": "train_1048576x128", "kind": "train", "m": 1 << 20, "n": 128, "b": 0, "kappa": 1e4, "rowmajor": True},
        # Page-locked host matrix in, host Q and R out.
        {"name": "host_262144x256", "kind": "host", "m": 1 << 18, "n": 256, "b": 64, "kappa": 1e5, "halving": False},
    ]


_MOST_FLOPS = 4.0 * (1 << 18) * 1024 * 1024  # the largest listed case


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _panels(rng, b_lo, b_hi, n_hi):
    """A width n = k b with a panel width b of any size, odd ones among them."""
    b = _log(rng, b_lo, b_hi)
    return b, b * rng.randint(1, max(1, min(8, n_hi // b)))


def draw(rng):
    kind = rng.choice(["factor", "factor", "option", "one_panel", "emulated", "batched", "graph", "train", "train_batch",
                       "host"])
    kappa = 10.0 ** rng.uniform(1, 5)
    rowmajor, keep = rng.random() < 0.5, rng.random() < 0.5
    if kind in ("factor", "option"):
        b, n = _panels(rng, 4, 160, 1024)
        m = max(_log(rng, 1000, 1 << 20), 2 * n)
        m = min(m, int(_MOST_FLOPS / (8.0 * n * n)))  # at most half the largest case
        case = {"kind": "factor", "m": m, "n": n, "b": b, "variant": rng.choice(["mcqr2gs", "mcqr2gs", "cqr2gs"]),
                "kappa": kappa, "rowmajor": rowmajor, "keep": keep}
        if kind == "option":
            case.update(variant="mcqr2gs", option=rng.choice(["lookahead", "adaptive", "halving"]))
        return case
    if kind == "one_panel":
        n = _log(rng, 8, 320)
        return {"kind": "factor", "m": max(_log(rng, 1000, 400000), 2 * n), "n": n, "b": 0,
                "variant": rng.choice(["cqr2", "scqr3"]), "kappa": kappa, "rowmajor": rowmajor, "keep": keep}
    if kind == "emulated":
        b, n = _panels(rng, 32, 160, 1024)
        return {"kind": "emulated", "m": _log(rng, 20000, 1 << 18), "n": n, "b": b, "kappa": kappa,
                "rowmajor": rowmajor, "keep": keep}
    if kind in ("batched", "graph"):
        big = kind == "batched"
        # n_step 0: widths 16, 32, 64, 128; else multiples of n_step up to 128 (2: widths that are no multiple of 4 too)
        return {"kind": kind, "count": rng.randint(4, 32), "m_lo": 2000 if big else 200,
                "m_hi": _log(rng, 20000, 200000) if big else _log(rng, 2000, 20000), "n_step": rng.choice([0, 0, 4, 2]),
                "shapes": rng.randint(1, 1 << 20), "k0": rng.choice([1, 2, 4]), "halving": False}
    if kind == "train":
        b, n = _panels(rng, 4, 128, 256)
        return {"kind": "train", "m": max(_log(rng, 1000, 1 << 20), 2 * n), "n": n, "b": b, "kappa": min(kappa, 1e4),
                "rowmajor": rowmajor}
    if kind == "train_batch":
        return {"kind": "train_batch", "count": rng.randint(2, 20), "m_lo": 10000, "m_hi": _log(rng, 20000, 100000),
                "n_step": 0, "shapes": rng.randint(1, 1 << 20), "k0": rng.choice([1, 2, 4])}
    b, n = _panels(rng, 8, 128, 512)
    return {"kind": "host", "m": max(_log(rng, 2000, 1 << 18), 2 * n), "n": n, "b": b, "kappa": kappa,
            "halving": rng.random() < 0.25}


# ------------------------------------------------------------------------------------------------- inputs
def _matrix(m, n, kappa, gen):
    """Column-major m x n on the GPU, condition number near kappa."""
    G = torch.randn((n, m), generator=gen, dtype=torch.float64, device="cuda").t()
    V = torch.linalg.qr(torch.randn((n, n), generator=gen, dtype=torch.float64, device="cuda")).Q
    s = torch.logspace(0, -math.log10(kappa), n, dtype=torch.float64, device="cuda") / math.sqrt(m)
    return (V @ (s[:, None] * G.t())).t()


def _shapes(case):
    """(m, n, b, kappa) of each matrix of a batch: part of the case, the same for every seed."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["count"]):
        m = int(rng.integers(case["m_lo"], case["m_hi"] + 1))
        if case["n_step"] == 0:
            n = int(rng.choice([16, 32, 64, 128]))
        else:
            n = case["n_step"] * int(rng.integers(8 // case["n_step"], 128 // case["n_step"] + 1))
        n = min(n, m // 2 // 4 * 4)
        k = case["k0"]
        while n % k or (n % 4 == 0 and (n // k) % 4):  # fewer panels where the width does not divide
            k -= 1
        out.append((m, n, n // k, 10.0 ** rng.uniform(1, 4)))
    return out


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return gen


def _inputs(case, seed):
    """The matrices of the case, and for a training step the upstream gradients of each Q and R."""
    gen = _generator(seed)
    if case["kind"] in ("batched", "graph", "train_batch"):
        As = [_matrix(m, n, kappa, gen) for m, n, _, kappa in _shapes(case)]
    else:
        As = [_matrix(case["m"], case["n"], case["kappa"], gen)]
    up = []
    if case["kind"] in ("train", "train_batch"):
        for A in As:
            m, n = A.shape
            up.append((torch.randn((m, n), generator=gen, dtype=torch.float64, device="cuda"),
                       torch.randn((n, n), generator=gen, dtype=torch.float64, device="cuda").triu()))
    return As, up


# ------------------------------------------------------------------------------------------------- a pass
def prepare(case, seed):
    As, up = _inputs(case, seed)
    kind = case["kind"]
    state = {"case": case, "kind": kind}
    if kind in ("factor", "emulated"):
        m, n, b = case["m"], case["n"], case["b"]
        A = As[0].contiguous() if case["rowmajor"] else As[0]
        opts = {"variant": case.get("variant", "mcqr2gs")}
        if kind == "emulated":
            opts["emulated"] = True
        if case.get("option"):
            opts[case["option"]] = True
        if case["keep"]:  # a loop that owns its buffers and stays asynchronous
            size = {k: v for k, v in opts.items() if k in ("variant", "emulated", "halving")}
            opts.update(out=(cqr.empty_colmajor(m, n, "cuda"), cqr.empty_colmajor(n, n, "cuda")), check=False,
                        workspace=torch.empty(cqr.workspace_size(m, n, b, **size), dtype=torch.uint8, device="cuda"))
        state.update(A=A, b=b, opts=opts)
    elif kind == "batched":
        state.update(As=As, bs=[b for _, _, b, _ in _shapes(case)], halving=case["halving"])
    elif kind == "graph":
        state["graph"] = cqr.BatchedGraph(As, [b for _, _, b, _ in _shapes(case)])
    elif kind == "train":
        A = As[0].contiguous() if case["rowmajor"] else As[0]
        state.update(A=A.requires_grad_(), b=case["b"], up=up[0])
    elif kind == "train_batch":
        state.update(As=[A.requires_grad_() for A in As], bs=[b for _, _, b, _ in _shapes(case)], up=up)
    else:
        m, n, b = case["m"], case["n"], case["b"]
        A = cqr.empty_colmajor_pinned(m, n)
        A.copy_(As[0])
        state.update(A=A, b=b, halving=case["halving"],
                     out=(cqr.empty_colmajor_pinned(m, n), cqr.empty_colmajor_pinned(n, n)),
                     dev=(cqr.empty_colmajor(m, n, "cuda"), cqr.empty_colmajor(n, n, "cuda")),
                     ws=torch.empty(cqr.workspace_size(m, n, b, halving=case["halving"]), dtype=torch.uint8,
                                    device="cuda"))
    return state


def run(state):
    kind = state["kind"]
    if kind in ("factor", "emulated"):
        return cqr.factor(state["A"], state["b"], **state["opts"])
    if kind == "batched":
        return cqr.factor_batched(state["As"], state["bs"], halving=state["halving"])
    if kind == "graph":
        return state["graph"].replay()
    if kind == "train":
        A = state["A"]
        A.grad = None
        Q, R = cqr.qr(A, state["b"])
        torch.autograd.backward([Q, R], list(state["up"]))
        return Q.detach(), R.detach(), A.grad
    if kind == "train_batch":
        for A in state["As"]:
            A.grad = None
        pairs = cqr.qr_batched(state["As"], state["bs"])
        torch.autograd.backward([t for p in pairs for t in p], [t for p in state["up"] for t in p])
        return [(Q.detach(), R.detach(), A.grad) for (Q, R), A in zip(pairs, state["As"])]
    return cqr.factor_host(state["A"], state["b"], out=state["out"], device_out=state["dev"], workspace=state["ws"],
                           halving=state["halving"])


# ------------------------------------------------------------------------------------------------- its measure
def work(case):
    """Each input read and each output written once; the method's multiply-adds (4 m n^2 for the two-pass methods,
    6 m n^2 for the three-pass one, 5 m n^2 for the adjoint)."""
    kind = case["kind"]
    if kind in ("batched", "graph", "train_batch"):
        sizes = [(m, n) for m, n, _, _ in _shapes(case)]
    else:
        sizes = [(case["m"], case["n"])]
    nbytes = flops = 0.0
    for m, n in sizes:
        nbytes += 8.0 * (2 * m * n + n * n)
        flops += (6.0 if case.get("variant") == "scqr3" else 4.0) * m * n * n
        if kind in ("train", "train_batch"):
            nbytes += 8.0 * (2 * m * n + n * n)  # dQ, dR in, the gradient out
            flops += 5.0 * m * n * n
    return {"bytes": nbytes, "flops": flops}


def _householder(A):
    """Householder QR with R's diagonal positive, as CholeskyQR has it."""
    Q, R = torch.linalg.qr(A)
    d = torch.where(torch.diagonal(R) < 0, -1.0, 1.0).to(R.dtype)
    return Q * d, d[:, None] * R


def exact(case, seed):
    As, up = _inputs(case, seed)
    kind = case["kind"]
    out = []
    for i, A in enumerate(As):
        if not up:
            out.append(_householder(A))
            continue
        dQ, dR = up[i]
        Q, R = _householder(A)
        M = R @ dR.t() - dQ.t() @ Q
        M = M.tril() + M.tril(-1).t()
        dA = torch.linalg.solve_triangular(R, (dQ + Q @ M).t(), upper=True).t()
        out.append((Q, R, dA))
    return out if kind in ("batched", "graph", "train_batch") else out[0]
