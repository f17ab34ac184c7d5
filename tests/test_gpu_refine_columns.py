"""Right-hand sides refined together: columns that stop at different times, groups, small workspaces."""
import ctypes

import pytest
import torch

from paper_1511_07174_gb300 import _lib, api, inputs

pytestmark = pytest.mark.gpu


def _case(n, k, seed):
    A = inputs.uniform(n, seed, "cuda")
    A.diagonal().add_(n ** 0.5)
    X = inputs.normal((n, k), seed + 1, "cuda")
    B = A @ X
    return A, B


@pytest.mark.parametrize("n,k,kw", [(70, 2, {}), (500, 4, {}), (1000, 5, dict(restart_m=3, restarts=4)), (333, 9, {})])
@pytest.mark.parametrize("zero", [None, 0, 1])
def test_columns_converge_on_their_own(n, k, kw, zero):
    A, B = _case(n, k, n + k)
    if zero is not None:
        B[:, zero] = 0.0  # done before the others begin
    F, ipiv, _ = api.lu_factor_mixed(A, "bf16")
    X, st = api.gmresir(A, F, ipiv, B, **kw)
    assert len(st) == k and all(s["converged"] for s in st)
    assert float(api.backward_error(A, X, B).max()) <= 1e-14
    if zero is not None:
        assert not bool(X[:, zero].any()) and st[zero]["outer"] == 0
    for c in range(k):
        x1, s1 = api.gmresir(A, F, ipiv, B[:, c].contiguous(), **kw)
        # the same iteration up to the rounding of the preconditioner
        assert s1["converged"] and abs(s1["outer"] - st[c]["outer"]) <= 1
        torch.testing.assert_close(X[:, c], x1, rtol=1e-9, atol=1e-11)


def test_smallest_workspace_and_step_limit():
    n, k = 400, 3
    A, B = _case(n, k, 5)
    Ac, Bc = api.colmajor(A), api.colmajor(B)
    F, ipiv, _ = api.lu_factor_mixed(A, "bf16")
    lib = _lib.load()
    X = api.colmajor(torch.empty_like(B))
    st = (_lib.GmresirStats * k)()

    def run(nbytes, max_outer):
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        opts = _lib.GmresirOpts(1e-14, 1e-8, max_outer, 50, 1)
        p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        return lib.gbla_gmresir_solve_nrhs(n, k, p(Ac), n, p(F), n, p(ipiv), p(Bc), n, p(X), n, ctypes.byref(opts), st,
                                           p(ws), nbytes, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))

    one = lib.gbla_gmresir_workspace(n, 50)
    assert run(one - 256, 10) == 1001
    for nbytes in (one, lib.gbla_gmresir_workspace_nrhs(n, 2, 50), lib.gbla_gmresir_workspace_nrhs(n, k, 50)):
        assert run(nbytes, 10) == 0 and all(s.converged for s in st)
        assert float(api.backward_error(A, X, B).max()) <= 1e-14
    # no step allowed: every column reports its first backward error
    assert run(one, 0) == _lib.GBLA_ERR_NOT_CONVERGED
    b1 = [s.beta0 for s in st]
    assert run(lib.gbla_gmresir_workspace_nrhs(n, k, 50), 0) == _lib.GBLA_ERR_NOT_CONVERGED
    assert not any(s.converged for s in st) and all(0.3 < s.beta0 / b < 3 for s, b in zip(st, b1))


# above 4096 rows the preconditioner runs with half the helper threads
@pytest.mark.parametrize("n,k", [(4160, 1), (4161, 3)])
def test_large_preconditioner(n, k):
    A, B = _case(n, k, 11)
    F, ipiv, _ = api.lu_factor_mixed(A, "bf16")
    X, st = api.gmresir(A, F, ipiv, B)
    assert all(s["converged"] for s in st) and float(api.backward_error(A, X, B).max()) <= 1e-14
