"""The steps inside an outer block: both tile sizes of the inner updates, narrow and wide substitutions."""
import pytest
import torch

from paper_1511_07174_gb300 import api, inputs

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def _perm(ipiv):
    p = list(range(len(ipiv)))
    for i, q in enumerate(ipiv.cpu().tolist()):
        p[i], p[q - 1] = p[q - 1], p[i]
    return torch.tensor(p, device="cuda")


# 5200 with nb = 256: the 64 x 64 tiles of the inner steps (304 of them from 4864 rows up)
@pytest.mark.parametrize("n,nb", [(33, 32), (65, 64), (129, 0), (300, 96), (257, 256), (1030, 160), (5200, 256)])
def test_lu_backward_error(n, nb):
    A = inputs.uniform(n, 100 + n, "cuda")
    LU, ipiv, info = api.lu_factor(A, nb=nb)
    L = torch.tril(LU, -1) + torch.eye(n, dtype=LU.dtype, device="cuda")
    U = torch.triu(LU)
    assert int(info.item()) == 0 and float(torch.tril(LU, -1).abs().max()) <= 1.0 + 2 * EPS
    # |P A - L U| <= gamma_n |L||U| (gamma_n = n u), and the residual's own rounding, as much again
    R = (A[_perm(ipiv)] - L @ U).abs() / (L.abs() @ U.abs())
    assert float(R.max()) <= 2 * n * EPS


# 7000 with nb = 256: the 64 x 64 tiles of the inner update (304 of them from 6528 rows up)
@pytest.mark.parametrize("n,nb", [(31, 64), (65, 64), (97, 0), (200, 128), (1025, 256), (7000, 256)])
def test_chol_backward_error(n, nb):
    A = inputs.spd_fp32_product(n, 200 + n, "cuda")
    F, info = api.chol_factor(A, nb=nb)
    L = torch.tril(F)
    assert int(info.item()) == 0
    R = torch.tril((A - L @ L.t()).abs() / (L.abs() @ L.abs().t()))
    assert float(R.max()) <= 2 * n * EPS


@pytest.mark.parametrize("n,nb", [(63, 64), (130, 128), (1100, 256)])
def test_chol_fp32_backward_error(n, nb):
    A = inputs.spd_fp32_product(n, 300 + n, "cuda")
    F, info = api.chol_factor_mixed(A, "fp32", nb=nb)
    L = torch.tril(F).double()
    assert int(info.item()) == 0
    R = torch.tril((A - L @ L.t()).abs() / (L.abs() @ L.abs().t()))
    assert float(R.max()) <= 2 * n * 2.0 ** -24
