"""Triangular solves: edges of blocks, chains and helper tasks; unsafe diagonal blocks; waits."""
import pytest
import torch

from paper_1511_07174_gb300 import api

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def _factors(n, seed):
    """LU as lu_factor stores it: |l| <= 1 with small off-diagonals, moderate pivots."""
    g = torch.Generator().manual_seed(seed)
    M = (torch.rand((n, n), generator=g, dtype=torch.float64) * 2 - 1) / max(1.0, n ** 0.5)
    M.diagonal().copy_(1.0 + torch.rand(n, generator=g, dtype=torch.float64))
    ipiv = torch.arange(1, n + 1, dtype=torch.int32)
    return M.cuda(), ipiv.cuda()


def _residual(M, X, B, trans):
    """max |B - op(LU) X| / (|L||U||X|), componentwise: <= c n u for a stable solve."""
    L = torch.tril(M, -1) + torch.eye(M.shape[0], dtype=M.dtype, device=M.device)
    U = torch.triu(M)
    if trans:
        L, U = U.t(), L.t()
    R = (B - L @ (U @ X)).abs()
    S = L.abs() @ (U.abs() @ X.abs())
    return float((R / S).max())


@pytest.mark.parametrize("n,nrhs", [(63, 2), (64, 1), (65, 1), (128, 3), (129, 4), (191, 5), (193, 1), (257, 8), (450, 9),
                                    (1088, 16), (1153, 17), (1216, 33), (2111, 1), (2500, 4)])
@pytest.mark.parametrize("trans", [False, True])
def test_solve_edges(n, nrhs, trans):
    M, ipiv = _factors(n, n + nrhs)
    g = torch.Generator().manual_seed(n)
    B = torch.randn((n, nrhs), generator=g, dtype=torch.float64).cuda()
    X = api.lu_solve(M, ipiv, B, trans=trans)
    # two substitutions of n terms each, blocks by their inverses, and the residual's own rounding
    assert _residual(M, X, B, trans) <= 8 * n * EPS


@pytest.mark.parametrize("n,nrhs", [(64, 1), (130, 4), (1100, 11)])
def test_chol_solve_edges(n, nrhs):
    M, _ = _factors(n, n)
    B = torch.randn((n, nrhs), dtype=torch.float64).cuda()
    X = api.chol_solve(M, B)
    L = torch.tril(M)
    R = (B - L @ (L.t() @ X)).abs()
    assert float((R / (L.abs() @ (L.t().abs() @ X.abs()))).max()) <= 8 * n * EPS


@pytest.mark.parametrize("trans", [False, True])
def test_result_does_not_depend_on_the_grid(trans):
    # one cluster alone: the chain's own CTAs do every task
    M, ipiv = _factors(2240, 3)
    B = torch.randn((2240, 3), dtype=torch.float64).cuda()
    X = api.lu_solve(M, ipiv, B, trans=trans)
    old = api.get_substitution_ctas()
    try:
        api.set_substitution_ctas(1)
        Y = api.lu_solve(M, ipiv, B, trans=trans)
        torch.cuda.synchronize()
    finally:
        api.set_substitution_ctas(old)
    assert torch.equal(X, Y)


def test_unsafe_diagonal_block_is_substituted():
    # the inverse of this block has elements of size 2^62; substitution solves it to working accuracy
    n = 320
    M, ipiv = _factors(n, 5)
    M[64:128, 64:128] = torch.tril(M[64:128, 64:128], -1) - torch.triu(torch.ones(64, 64, dtype=M.dtype, device=M.device), 1) \
        + torch.eye(64, dtype=M.dtype, device=M.device)
    B = torch.randn((n, 2), dtype=torch.float64).cuda()
    X = api.lu_solve(M, ipiv, B)
    assert _residual(M, X, B, False) <= 8 * n * EPS


@pytest.mark.parametrize("trans", [False, True])
def test_badly_conditioned_diagonal_block_is_refined(trans):
    # the inverse of this block has elements of size 1.25^62 (about 1e6)
    n = 320
    M, ipiv = _factors(n, 6)
    M[64:128, 64:128] = torch.tril(M[64:128, 64:128], -1) - 0.25 * torch.triu(torch.ones(64, 64, dtype=M.dtype, device=M.device), 1) \
        + torch.eye(64, dtype=M.dtype, device=M.device)
    X = torch.randn((n, 3), dtype=torch.float64).cuda()
    L = torch.tril(M, -1) + torch.eye(n, dtype=M.dtype, device=M.device)
    B = torch.triu(M).t() @ (L.t() @ X) if trans else L @ (torch.triu(M) @ X)
    X = api.lu_solve(M, ipiv, B, trans=trans)
    assert _residual(M, X, B, trans) <= 8 * n * EPS


def test_zero_pivot_and_nan_follow_ieee():
    n = 200
    M, ipiv = _factors(n, 7)
    B = torch.randn((n, 1), dtype=torch.float64).cuda()
    Bn = B.clone()
    Bn[150] = torch.full((1,), -1, dtype=torch.int64).view(torch.float64).item()  # NaN, all bits set
    X = api.lu_solve(M, ipiv, Bn)
    assert bool(torch.isnan(X).all())  # U couples every row above 150, L every row below
    M[199, 199] = 0.0
    X = api.lu_solve(M, ipiv, B)
    assert not bool(torch.isfinite(X).any())


def test_wait_limit_reports_status():
    M, ipiv = _factors(1500, 9)
    B = torch.randn((1500, 2), dtype=torch.float64).cuda()
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    old = api.get_wait_timeout_ns()
    try:
        api.set_wait_timeout_ns(0)
        api.lu_solve(M, ipiv, B, info=info)
        torch.cuda.synchronize()
        assert int(info.item()) != 0
    finally:
        api.set_wait_timeout_ns(old)
    X = api.lu_solve(M, ipiv, B, info=info)
    assert int(info.item()) == 0 and _residual(M, X, B, False) <= 8 * 1500 * EPS
