"""Rows below a Cholesky diagonal block: the first 32 columns' part of an element is summed before it is subtracted."""
import pytest
import torch

from paper_1511_07174_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("below", [1, 40])
def test_small_terms_are_not_lost_one_by_one(below):
    # L11 = [[I, 0], [2^-27, I]] in halves of 32, the rows below [2^-27 .., 1 - 2^-49 ..]: each of the 32
    # products 2^-54 vanishes next to 1, their sum 2^-49 does not
    n, e = 64 + below, 2.0 ** -27
    A = torch.eye(n, dtype=torch.float64)
    A[32:64, :32] = e
    A[32:64, 32:64] += 32 * e * e * (1 - torch.eye(32, dtype=torch.float64))
    A[64:, :32], A[64:, 32:64] = e, 1.0
    A[64:, 64:] += 33.0
    A = torch.tril(A) + torch.tril(A, -1).t()
    A[64:, 64:] += 100.0 * torch.eye(below, dtype=torch.float64)
    F, info = api.chol_factor(A.cuda())
    F = F.cpu()
    assert int(info.item()) == 0
    assert torch.equal(torch.tril(F[:64, :64]), torch.tril(torch.eye(64, dtype=torch.float64) + torch.nn.functional.pad(
        torch.full((32, 32), e, dtype=torch.float64), (0, 32, 32, 0))))
    assert torch.equal(F[64:, 32:64], torch.full((below, 32), 1.0 - 2.0 ** -49, dtype=torch.float64))
