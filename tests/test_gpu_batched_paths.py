"""Batched LU / Cholesky: the panel path against the column-by-column path, bit for bit.

Both apply the same operations to every element in the same order, so for any order,
type and number of right-hand sides the factors, pivots, info words and solutions are
identical. Orders at the edges of the 16-column panels, the 32-row tiles, one and two
rows per thread and the largest order the panels take; max_n below an order sends that
system to the column-by-column path, in the middle of a batch of both.
"""
import pytest
import torch

from paper_1511_07174_gb300.batched import BatchedLU

pytestmark = pytest.mark.gpu

EDGES = {128: [1, 2, 15, 16, 17, 31, 32, 33, 48, 63, 127, 128],
         256: [5, 16, 129, 144, 161, 240, 255, 256],
         520: [3, 17, 257, 272, 300, 383, 496, 511, 512, 513, 520]}


def _systems(sizes, method, singular):
    g = torch.Generator().manual_seed(sum(sizes))
    As, Bs = [], []
    for i, n in enumerate(sizes):
        A = torch.rand((n, n), generator=g, dtype=torch.float64) * 2 - 1
        if method == "chol":
            A = A @ A.t() / n + torch.eye(n, dtype=torch.float64)
            if singular and i % 3 == 2:
                A[n // 2, n // 2] = -1.0      # stops in the middle
        elif singular and i % 3 == 2:
            A[:, n // 2] = 0.0                # a zero pivot: the elimination goes on
        As.append(A)
        Bs.append(torch.randn((n, 1 + i % 4), generator=g, dtype=torch.float64))
    return As, Bs


@pytest.mark.parametrize("method", ["lu", "chol"])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("top", sorted(EDGES))
@pytest.mark.parametrize("singular", [False, True])
def test_panel_path_is_the_column_path(method, dtype, top, singular):
    As, Bs = _systems(EDGES[top], method, singular)
    runs = []
    for max_n in (top, 8):  # 8: everything above 32 rows goes column by column
        bl = BatchedLU(As, Bs, dtype=dtype, method=method)
        bl.max_n = max_n
        bl.restore()
        bl.run()
        torch.cuda.synchronize()
        runs.append(bl)
    a, b = runs
    assert torch.equal(a.info, b.info)
    if method == "lu":
        assert torch.equal(a.ipiv, b.ipiv)
        torch.testing.assert_close(a.A, b.A, rtol=0, atol=0, equal_nan=True)
        torch.testing.assert_close(a.B, b.B, rtol=0, atol=0, equal_nan=True)
    else:
        # the panels' FP64 reciprocal root is rounded once, the column path's twice
        tol = 0.0 if dtype == torch.float32 else 600 * 2.0 ** -52
        torch.testing.assert_close(a.A, b.A, rtol=tol, atol=tol)
        torch.testing.assert_close(a.B, b.B, rtol=100 * tol, atol=100 * tol)
    assert bool((a.info != 0).any()) == singular


def test_nan_column_is_no_interchange():
    """A column of NaN offers no pivot: the call ends, its pivot is the row itself."""
    As, Bs = _systems([40, 200], "lu", False)
    As[1][:, 70] = float("nan")
    bl = BatchedLU(As, Bs)
    bl.restore()
    bl.run()
    torch.cuda.synchronize()
    piv = bl.ipiv.cpu()
    assert int(piv[40 + 70]) == 71
    assert torch.isfinite(bl.B[:40]).all()
