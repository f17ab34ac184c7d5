"""A right-hand side's solution does not depend on the others that are solved or refined with it: bit for bit."""
import ctypes

import pytest
import torch

from paper_1511_07174_gb300 import _lib, api, inputs

pytestmark = pytest.mark.gpu


def _case(n, k):
    A = inputs.uniform(n, n, "cuda")
    A.diagonal().add_(n ** 0.5)
    return A, inputs.normal((n, k), n + 1, "cuda")


@pytest.mark.parametrize("n,k", [(64, 5), (130, 4), (400, 7), (1100, 17), (1500, 2)])
def test_solve(n, k):
    A, B = _case(n, k)
    LU, ipiv, _ = api.lu_factor(inputs.uniform(n, 3, "cuda"))  # blocks that are refined among them
    F, _ = api.chol_factor(inputs.spd_fp32_product(n, 4, "cuda"))
    for c in range(0, k, 3):
        b = B[:, c:c + 1].contiguous()
        for trans in (False, True):
            assert torch.equal(api.lu_solve(LU, ipiv, B, trans=trans)[:, c:c + 1], api.lu_solve(LU, ipiv, b, trans=trans))
        assert torch.equal(api.chol_solve(F, B)[:, c:c + 1], api.chol_solve(F, b))


# 4200: the preconditioner's variant of large systems
@pytest.mark.parametrize("n,k,kw", [(70, 2, {}), (500, 4, {}), (1000, 5, dict(restart_m=3, restarts=4)), (4200, 3, {})])
def test_refinement(n, k, kw):
    A, B = _case(n, k)
    F, ipiv, _ = api.lu_factor_mixed(A, "bf16")
    X, st = api.gmresir(A, F, ipiv, B, **kw)
    for c in range(k):
        x1, s1 = api.gmresir(A, F, ipiv, B[:, c].contiguous(), **kw)
        assert torch.equal(X[:, c], x1) and s1 == st[c]


def test_refinement_with_less_scratch():
    n, k = 300, 3
    A, B = _case(n, k)
    Ac, Bc = api.colmajor(A), api.colmajor(B)
    F, ipiv, _ = api.lu_factor_mixed(A, "bf16")
    lib = _lib.load()
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    out = []
    for cols in (1, 2, 3):
        X = api.colmajor(torch.zeros_like(B))
        ws = torch.empty(lib.gbla_gmresir_workspace_nrhs(n, cols, 50), dtype=torch.uint8, device="cuda")
        st = (_lib.GmresirStats * k)()
        assert lib.gbla_gmresir_solve_nrhs(n, k, p(Ac), n, p(F), n, p(ipiv), p(Bc), n, p(X), n,
                                           ctypes.byref(_lib.GmresirOpts(1e-14, 1e-8, 10, 50, 1)), st, p(ws), ws.numel(),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        out.append(X)
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
