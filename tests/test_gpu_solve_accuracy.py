"""Solves of small systems are as accurate as a substitution."""
import numpy as np
import pytest
import torch

import oracle
from paper_1511_07174_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _exact(LU, b):
    """L U x = b in extended precision."""
    n = len(b)
    M, x = LU.astype(np.longdouble), b.astype(np.longdouble)
    for i in range(n):
        x[i + 1:] -= M[i + 1:, i] * x[i]
    for i in range(n - 1, -1, -1):
        x[i] /= M[i, i]
        x[:i] -= M[:i, i] * x[i]
    return x


@pytest.mark.parametrize("n", [100, 200])
def test_error_is_not_larger_than_a_substitution_s(n):
    ident = np.arange(1, n + 1, dtype=np.int32)
    ratios = []
    for seed in range(24):
        LU, _, _ = oracle.getrf(np.asfortranarray(inputs.uniform(n, seed=1000 + seed).numpy()))
        b = np.random.default_rng(seed).standard_normal(n)
        x = _exact(LU, b)
        X = api.lu_solve(torch.from_numpy(LU).cuda(), torch.from_numpy(ident).cuda(), torch.from_numpy(b).cuda().unsqueeze(1))
        err = lambda y: float(np.sqrt(((y - x) ** 2).sum()))  # noqa: E731
        ratios.append(err(X.cpu().numpy()[:, 0]) / err(np.asarray(oracle.getrs(LU, ident, b.reshape(-1, 1))).reshape(-1)))
    # 24 errors against 24 errors of the plain FP64 substitution
    assert float(np.exp(np.mean(np.log(ratios)))) <= 1.0
