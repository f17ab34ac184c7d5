"""What a user of this library has it do, as cases that can be timed and compared.

Each case is one pass through the public entry points (`api`, `batched`): FP64 LU and
Cholesky with their solves, the differentiable solve, batches of small systems, the
mixed-precision solvers refined to FP64 accuracy, and the standalone Krylov solvers.
`listed` holds the cases themselves, `draw` gives more of the same ranges, `prepare`
makes what a program has in hand before the call (on the GPU, from the seed alone),
`run` is the pass, `work` what it cannot do without, and `exact` what plain torch gives
for the same inputs in 64 bits.
"""
import math

import torch

from paper_1511_07174_gb300 import api, inputs
from paper_1511_07174_gb300.batched import BatchedLU

DEV = "cuda"


def listed():
    return [
        # The smallest call of the library's workloads: one dense system of order 512, one
        # right-hand side, factored and solved once. Latency and launches are all that counts.
        {"name": "lu_n512", "kind": "lu", "n": 512, "nrhs": 1},
        # An ordinary FP64 solve at a ragged size with a few right-hand sides.
        {"name": "lu_n3001_rhs3", "kind": "lu", "n": 3001, "nrhs": 3},
        # The large FP64 LU with 16 right-hand sides (the FP64 reference of the benchmark).
        {"name": "lu_n8192_rhs16", "kind": "lu", "n": 8192, "nrhs": 16},
        # Factors kept, new right-hand sides arriving: a solve with A and one with A^t.
        {"name": "resolve_n4096_rhs16", "kind": "resolve", "n": 4096, "nrhs": 16},
        # SPD system (a Gram matrix plus the identity) in FP64, default block size, ragged size.
        {"name": "chol_n6000_rhs4", "kind": "chol", "n": 6000, "nrhs": 4},
        # The differentiable solve inside a training loop: forward and backward.
        {"name": "grad_n4096_rhs8", "kind": "grad", "n": 4096, "nrhs": 8, "method": "lu"},
        # Thousands of small systems of uneven size at once, factored and solved, in FP64 and
        # FP32, and the SPD counterpart.
        {"name": "batched_lu_fp64", "kind": "batched", "batch": 4096, "nmin": 16, "nmax": 256,
         "dtype": "float64", "method": "lu"},
        {"name": "batched_lu_fp32", "kind": "batched", "batch": 4096, "nmin": 16, "nmax": 256,
         "dtype": "float32", "method": "lu"},
        {"name": "batched_chol_fp64", "kind": "batched", "batch": 2048, "nmin": 16, "nmax": 256,
         "dtype": "float64", "method": "chol"},
        # The headline: one large system solved in mixed precision and refined by GMRES to FP64
        # accuracy (half-precision products split in three, condition number 1e4).
        {"name": "mixed_n16384_fp16x3", "kind": "mixed", "n": 16384, "nrhs": 1, "prec": "fp16x3",
         "kappa": 1e4},
        # A middle-sized well-conditioned system, plain bf16 update, several right-hand sides
        # refined from the same factors, ragged size.
        {"name": "mixed_n2500_bf16_rhs4", "kind": "mixed", "n": 2500, "nrhs": 4, "prec": "bf16",
         "kappa": 1e2},
        # The SPD counterpart of the mixed-precision solve.
        {"name": "chol_mixed_n8192", "kind": "chol_mixed", "n": 8192, "nrhs": 1, "prec": "fp16x3"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lu", "lu", "resolve", "chol", "grad", "batched", "batched", "mixed", "mixed",
                       "chol_mixed", "krylov"])
    if kind in ("lu", "resolve", "chol"):
        return {"kind": kind, "n": _log_int(rng, 48, 8192), "nrhs": rng.randint(1, 24)}
    if kind == "grad":
        return {"kind": kind, "n": _log_int(rng, 96, 4096), "nrhs": rng.randint(1, 16),
                "method": rng.choice(["lu", "chol"])}
    if kind == "batched":
        nmin = rng.randint(4, 64)
        return {"kind": kind, "batch": _log_int(rng, 64, 4096), "nmin": nmin,
                "nmax": rng.randint(nmin + 16, 256), "dtype": rng.choice(["float64", "float32"]),
                "method": rng.choice(["lu", "chol"])}
    if kind == "mixed":
        prec = rng.choice(["fp16x3", "fp16x3", "bf16x3", "fp32", "bf16", "fp16", "tf32"])
        split = prec in ("fp16x3", "bf16x3", "fp32")
        return {"kind": kind, "n": _log_int(rng, 500, 16384 if split else 4096),
                "nrhs": rng.randint(1, 4), "prec": prec, "kappa": 1e4 if prec in ("fp16x3", "fp32") else 1e2}
    if kind == "chol_mixed":
        return {"kind": kind, "n": _log_int(rng, 500, 16384), "nrhs": rng.randint(1, 4),
                "prec": rng.choice(["fp16x3", "bf16x3", "fp16", "bf16"])}
    return {"kind": kind, "n": _log_int(rng, 300, 8192), "solver": rng.choice(["gmres", "bicgstab"])}


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _mix_rows(M, g):
    """Q M with Q a random orthogonal matrix applied in O(n log n) per column: twice,
    random signs and then the (orthonormal, symmetric) Hartley transform."""
    n = M.shape[0]
    for _ in range(2):
        signs = (torch.randint(0, 2, (n, 1), generator=g, device=DEV) * 2 - 1).to(M.dtype)
        for c in range(0, M.shape[1], 2048):
            F = torch.fft.fft(M[:, c:c + 2048] * signs, dim=0)
            M[:, c:c + 2048] = (F.real - F.imag) / math.sqrt(n)
    return M


def _spectrum_matrix(n, kappa, seed):
    """Dense A = Q1 diag(s) Q2^t with singular values spaced geometrically from 1 to 1/kappa."""
    g = _gen(seed)
    s = inputs.kappa_spectrum(n, kappa, DEV)[torch.randperm(n, generator=g, device=DEV)]
    M = _mix_rows(torch.diag(s), g)
    return _mix_rows(M.t().contiguous(), g)


def _system(case, seed):
    """(A, B) of a dense case."""
    n, kind = case["n"], case["kind"]
    if kind in ("chol", "chol_mixed") or case.get("method") == "chol":
        A = inputs.spd_fp32_product(n, seed, DEV)
    elif kind == "mixed":
        A = _spectrum_matrix(n, case["kappa"], seed)
    elif kind in ("grad", "krylov"):
        A = inputs.uniform(n, seed, DEV)
        A.diagonal().add_(math.sqrt(n))
    else:
        A = inputs.uniform(n, seed, DEV)
    B = A @ inputs.normal((n, case.get("nrhs", 1)), seed + 1, DEV)
    return A, B


def _batch(case, seed):
    """Systems of uneven size: sizes uniform in [nmin, nmax], 1 to 4 right-hand sides each
    (the case's own sizes, whatever the seed), A = U[-1, 1] + n I (LU) or a Gram matrix / n + I
    (Cholesky)."""
    g = torch.Generator().manual_seed(case["batch"] * 1000 + case["nmax"])
    sizes = torch.randint(case["nmin"], case["nmax"] + 1, (case["batch"],), generator=g).tolist()
    nrhs = torch.randint(1, 5, (case["batch"],), generator=g).tolist()
    dtype = getattr(torch, case["dtype"])
    gd = _gen(seed)
    As, Bs = [], []
    for n0 in range(0, case["batch"], 512):
        ns, ks = sizes[n0:n0 + 512], nrhs[n0:n0 + 512]
        flat = torch.rand(sum(n * n for n in ns), generator=gd, dtype=torch.float64, device=DEV) * 2 - 1
        b = torch.randn(sum(n * k for n, k in zip(ns, ks)), generator=gd, dtype=torch.float64, device=DEV)
        mats = [m.view(n, n) for m, n in zip(flat.split([n * n for n in ns]), ns)]
        if case["method"] == "chol":
            mats = [m @ m.t() / n for m, n in zip(mats, ns)]
        for m, n in zip(mats, ns):
            m.diagonal().add_(1.0 if case["method"] == "chol" else float(n))
        As += [m.to(dtype) for m in mats]
        Bs += [v.view(n, k).to(dtype) for v, n, k in zip(b.split([n * k for n, k in zip(ns, ks)]), ns, ks)]
    return As, Bs


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batched":
        As, Bs = _batch(case, seed)
        return {"case": case, "bl": BatchedLU(As, Bs, dtype=getattr(torch, case["dtype"]), device=DEV,
                                              method=case["method"])}
    A, B = _system(case, seed)
    st = {"case": case, "A": A, "B": B}
    if kind == "resolve":
        st["LU"], st["ipiv"], _ = api.lu_factor(A)
    elif kind == "grad":
        A.requires_grad_()
        B.requires_grad_()
        st["g"] = inputs.normal(tuple(B.shape), seed + 2, DEV)
    elif kind in ("mixed", "chol_mixed", "krylov") and B.shape[1] == 1:
        st["B"] = B[:, 0].contiguous()
    return st


# -------------------------------------------------------------------------------- pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batched":
        bl = state["bl"]
        bl.restore()
        bl.run()
        out = {"A": bl.A, "X": bl.B, "info": bl.info}
        if case["method"] == "lu":
            out["ipiv"] = bl.ipiv
        return out
    A, B = state["A"], state["B"]
    if kind == "lu":
        LU, ipiv, info = api.lu_factor(A)
        return {"LU": LU, "ipiv": ipiv, "info": info, "X": api.lu_solve(LU, ipiv, B)}
    if kind == "resolve":
        return {"X": api.lu_solve(state["LU"], state["ipiv"], B),
                "Xt": api.lu_solve(state["LU"], state["ipiv"], B, trans=True)}
    if kind == "chol":
        F, info = api.chol_factor(A)
        return {"F": F, "info": info, "X": api.chol_solve(F, B)}
    if kind == "grad":
        x = api.solve(A, B, method=case["method"])
        gA, gB = torch.autograd.grad(x, (A, B), state["g"])
        return {"x": x.detach(), "gA": gA, "gB": gB}
    if kind == "mixed":
        return {"x": api.solve_mixed(A, B, prec=case["prec"])[0]}
    if kind == "chol_mixed":
        return {"x": api.solve_chol_mixed(A, B, prec=case["prec"])[0]}
    solver = api.gmres if case["solver"] == "gmres" else api.bicgstab
    return {"x": solver(A, B, tol=1e-12)[0]}


# -------------------------------------------------------------------------------- work
def _sizes(case):
    """Sizes and right-hand sides of a batch, from their expectations (uniform draws)."""
    a, b = case["nmin"], case["nmax"]
    m = b - a + 1
    n2 = sum(n * n for n in range(a, b + 1)) / m
    n3 = sum(n ** 3 for n in range(a, b + 1)) / m
    return (a + b) / 2.0, n2, n3


def work(case):
    kind = case["kind"]
    if kind == "batched":
        es = 8 if case["dtype"] == "float64" else 4
        n1, n2, n3 = _sizes(case)
        f = 2.0 / 3.0 if case["method"] == "lu" else 1.0 / 3.0
        return {"bytes": case["batch"] * es * (2 * n2 + 2 * 2.5 * n1),
                "flops": case["batch"] * (f * n3 + 2 * 2.5 * n2)}
    n, k = case["n"], case.get("nrhs", 1)
    if kind == "lu":
        return {"bytes": 16.0 * n * n + 16.0 * n * k, "flops": 2.0 / 3.0 * n ** 3 + 2.0 * n * n * k}
    if kind == "resolve":
        return {"bytes": 8.0 * n * n + 24.0 * n * k, "flops": 4.0 * n * n * k}
    if kind == "chol":
        return {"bytes": 16.0 * n * n + 16.0 * n * k, "flops": 1.0 / 3.0 * n ** 3 + 2.0 * n * n * k}
    if kind == "grad":
        f = 2.0 / 3.0 if case["method"] == "lu" else 1.0 / 3.0
        return {"bytes": 16.0 * n * n + 32.0 * n * k, "flops": f * n ** 3 + 6.0 * n * n * k}
    if kind in ("mixed", "chol_mixed"):
        f = 2.0 / 3.0 if kind == "mixed" else 1.0 / 3.0
        return {"bytes": 8.0 * n * n + 16.0 * n * k, "flops": f * n ** 3 + 4.0 * n * n * k}
    return {"bytes": 8.0 * n * n + 16.0 * n, "flops": 40.0 * n * n}  # some 20 products with A


# ------------------------------------------------------------------------------- exact
def _exact_batched(case, seed):
    """LAPACK-style factors of the whole batch at once: every system padded with the
    identity to the largest order, which leaves its own factors and pivots as they are."""
    As, Bs = _batch(case, seed)
    nmax = max(A.shape[0] for A in As)
    fa, fb = [], []
    for c in range(0, len(As), 512):
        a, b = As[c:c + 512], Bs[c:c + 512]
        P = torch.eye(nmax, dtype=torch.float64, device=DEV).repeat(len(a), 1, 1)
        R = torch.zeros(len(a), nmax, 4, dtype=torch.float64, device=DEV)
        for i, (A, B) in enumerate(zip(a, b)):
            P[i, :A.shape[0], :A.shape[0]] = A
            R[i, :B.shape[0], :B.shape[1]] = B
        if case["method"] == "lu":
            F, piv = torch.linalg.lu_factor(P)
            X = torch.linalg.lu_solve(F, piv, R)
        else:
            L = torch.linalg.cholesky(P)
            X = torch.cholesky_solve(R, L)
            F = torch.tril(L) + torch.triu(P, 1)
        for i, (A, B) in enumerate(zip(a, b)):
            fa.append(F[i, :A.shape[0], :A.shape[0]].t().reshape(-1))
            fb.append(X[i, :B.shape[0], :B.shape[1]].t().reshape(-1))
    out = {"A": torch.cat(fa), "X": torch.cat(fb), "info": None}
    if case["method"] == "lu":
        out["ipiv"] = None
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batched":
        return _exact_batched(case, seed)
    A, B = _system(case, seed)
    if kind == "lu":
        LU, piv = torch.linalg.lu_factor(A)
        return {"LU": LU, "ipiv": None, "info": None, "X": torch.linalg.lu_solve(LU, piv, B)}
    if kind == "resolve":
        LU, piv = torch.linalg.lu_factor(A)
        return {"X": torch.linalg.lu_solve(LU, piv, B),
                "Xt": torch.linalg.lu_solve(LU, piv, B, adjoint=True)}
    if kind == "chol":
        L = torch.linalg.cholesky(A)
        return {"F": torch.tril(L) + torch.triu(A, 1), "info": None, "X": torch.cholesky_solve(B, L)}
    if kind == "grad":
        g = inputs.normal(tuple(B.shape), seed + 2, DEV)
        LU, piv = torch.linalg.lu_factor(A)
        x = torch.linalg.lu_solve(LU, piv, B)
        gB = torch.linalg.lu_solve(LU, piv, g, adjoint=True)
        return {"x": x, "gA": -gB @ x.t(), "gB": gB}
    x = torch.linalg.solve(A, B)
    return {"x": x[:, 0] if B.shape[1] == 1 else x}
