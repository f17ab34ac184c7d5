"""Solves of one 64-row block: groups of columns; permutations of one and two chunks of pivots."""
import numpy as np
import pytest
import torch

import oracle
from paper_1511_07174_gb300 import api, inputs

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("n,nrhs", [(1, 1), (1, 33), (33, 31), (33, 32), (64, 33), (64, 65), (40, 130), (255, 2), (256, 3), (257, 1)])
@pytest.mark.parametrize("trans", [False, True])
def test_small_solve(n, nrhs, trans):
    A = inputs.uniform(n, seed=60 + n)
    LU, ipiv, _ = oracle.getrf(np.asfortranarray(A.numpy()))
    B = torch.randn((n, nrhs), generator=torch.Generator().manual_seed(n), dtype=torch.float64)
    X = api.lu_solve(torch.from_numpy(LU).cuda(), torch.from_numpy(np.asarray(ipiv)).cuda(), B.cuda(), trans=trans).cpu()
    L, Uf = oracle.unpack_lu(LU)
    P = torch.from_numpy(np.asarray(oracle.perm_from_ipiv(ipiv, n)).astype(np.int64))
    M = torch.from_numpy(L @ Uf)
    G = torch.from_numpy(np.abs(L) @ np.abs(Uf))
    # P A = L U: componentwise residual of two substitutions and of the product here, 3 n u each at most
    if trans:
        R = (B - M.t() @ X[P]).abs() / (G.t() @ X[P].abs())
    else:
        R = (B[P] - M @ X).abs() / (G @ X.abs())
    assert float(R.max()) <= 9 * n * U


@pytest.mark.parametrize("nrhs", [32, 65])
def test_small_chol_solve(nrhs):
    n = 50
    F, _ = oracle.potrf(np.asfortranarray(inputs.spd(n, seed=4).numpy()))
    L = torch.from_numpy(np.tril(F))
    B = torch.randn((n, nrhs), generator=torch.Generator().manual_seed(1), dtype=torch.float64)
    X = api.chol_solve(torch.from_numpy(F).cuda(), B.cuda()).cpu()
    R = (B - L @ (L.t() @ X)).abs() / (L.abs() @ (L.t().abs() @ X.abs()))
    assert float(R.max()) <= 9 * n * U
