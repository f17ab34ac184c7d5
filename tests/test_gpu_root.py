"""Cholesky's root and the reciprocal its column is scaled with: those of sqrt and division, bit for bit."""
import pytest
import torch

from paper_1511_07174_gb300 import api
from paper_1511_07174_gb300.batched import BatchedLU

pytestmark = pytest.mark.gpu


def _diagonals(n):
    g = torch.Generator().manual_seed(11)
    ex = torch.randint(-2, 2, (n,), generator=g)
    ex[n // 2:] = torch.randint(-1000, 1000, (n - n // 2,), generator=g)
    d = torch.ldexp(torch.rand(n, generator=g, dtype=torch.float64) + 1.0, ex)
    d[:4] = torch.tensor([1.0, 4.0, 2.0 - 2.0 ** -52, 2.0 ** -1060], dtype=torch.float64)  # the last: subnormal
    return d


def test_batched():
    d = _diagonals(20000)
    As = [torch.tensor([[v, 1.0], [1.0, 4.0 / v]], dtype=torch.float64) for v in d.tolist()]
    bl = BatchedLU(As, method="chol")
    bl.restore()
    bl.run()
    F = bl.A.cpu().reshape(-1, 4)
    assert torch.equal(F[:, 0], d.sqrt())
    assert torch.equal(F[:, 1], 1.0 / d.sqrt())  # l_10 = 1 times the reciprocal


def test_diagonal_block():
    # the order-2 systems along the diagonal of one matrix: every 64-row block has 32 of them
    d = _diagonals(2000)[4:]
    n = 2 * d.numel()
    A = torch.zeros((n, n), dtype=torch.float64)
    i = torch.arange(0, n, 2)
    A[i, i], A[i + 1, i], A[i, i + 1], A[i + 1, i + 1] = d, torch.ones_like(d), torch.ones_like(d), 4.0 / d
    F, info = api.chol_factor(A.cuda())
    F = F.cpu()
    assert int(info.item()) == 0
    assert torch.equal(F[i, i], d.sqrt()) and torch.equal(F[i + 1, i], 1.0 / d.sqrt())
