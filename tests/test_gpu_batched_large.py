"""Batches with orders above 512, which are eliminated in place: the launch shape changes the time, not the result."""
import pytest
import torch

from paper_1511_07174_gb300.batched import BatchedLU

pytestmark = pytest.mark.gpu


def _systems(sizes, method):
    g = torch.Generator().manual_seed(sum(sizes))
    As, Bs = [], []
    for i, n in enumerate(sizes):
        A = torch.rand((n, n), generator=g, dtype=torch.float64) * 2 - 1
        if method == "chol":
            A = A @ A.t() / n + torch.eye(n, dtype=torch.float64)
        As.append(A)
        Bs.append(torch.randn((n, 1 + i % 4), generator=g, dtype=torch.float64))
    return As, Bs


@pytest.mark.parametrize("method", ["lu", "chol"])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_shape_does_not_change_the_result(method, dtype):
    # one row short of and past the panels' 512, the 128-row steps of the update, small systems beside them
    As, Bs = _systems([3, 40, 300, 511, 512, 513, 545, 640, 641], method)
    ref = None
    for threads, ctas in ((256, 0), (512, 1), (512, 2), (1024, 1), (1024, 4)):
        bl = BatchedLU(As, Bs, dtype=dtype, method=method)
        bl.restore()
        bl.run(threads, ctas)
        torch.cuda.synchronize()
        assert not bool(bl.info.any())
        if ref is None:
            ref = bl
        elif method == "lu":
            assert torch.equal(bl.A, ref.A) and torch.equal(bl.B, ref.B) and torch.equal(bl.ipiv, ref.ipiv)
        else:
            # fewer rows fit the panels, whose FP64 reciprocal root is rounded once, the column path's twice
            tol = 0.0 if dtype == torch.float32 else 600 * 2.0 ** -52
            torch.testing.assert_close(bl.A, ref.A, rtol=tol, atol=tol)
            torch.testing.assert_close(bl.B, ref.B, rtol=100 * tol, atol=100 * tol)
