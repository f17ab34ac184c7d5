"""The growth of an inverted diagonal block is that of its whole rows, not of 16 columns of them."""
import numpy as np
import pytest
import torch

from paper_1511_07174_gb300 import api

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _block(seed):
    """(T, x): upper triangular with the growth of its rows, sum_c |T^-1|_rc (|T| 1)_c, above 1024, where
    blocks are refined, and below it on any 16 columns; T x does not cancel, T^-1 (T x) does."""
    rng = np.random.default_rng(seed)
    T = np.eye(64) + np.triu(rng.random((64, 64)), 1)
    x = 0.5 + rng.random(64)
    parts = (np.abs(np.linalg.inv(T)) * np.abs(T).sum(1)).reshape(64, 4, 16).sum(2)
    assert parts.max() < 1000 and parts.sum(1).max() > 1100
    return T, x


@pytest.mark.parametrize("seed", [1, 2])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_growth_spread_over_all_columns_is_refined(seed, nrhs):
    T, x = _block(seed)
    n = 192
    M = torch.eye(n, dtype=torch.float64)
    M[64:128, 64:128] = torch.from_numpy(T)
    B = torch.ones((n, nrhs), dtype=torch.float64)
    B[64:128] = torch.from_numpy(T @ x).unsqueeze(1)
    X = api.lu_solve(M.cuda(), torch.arange(1, n + 1, dtype=torch.int32).cuda(), B.cuda()).cpu().numpy()
    assert np.array_equal(X[:64], B[:64].numpy()) and np.array_equal(X[128:], B[128:].numpy())
    Tl = T.astype(np.longdouble)
    for c in range(nrhs):
        xc = X[64:128, c].astype(np.longdouble)
        r = np.abs(B[64:128, c].numpy().astype(np.longdouble) - Tl @ xc) / (Tl @ np.abs(xc))
        # a refined block: the rounding of x (u) and that of the residual it was refined with (a sum of
        # 64 terms, some 4 u); D y alone: 25 u and 50 u in a model of it
        assert float(r.max()) <= 6 * U
