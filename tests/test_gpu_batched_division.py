"""The quotients of the batched substitutions are those of a division, whatever the exponents."""
import pytest
import torch

from paper_1511_07174_gb300.batched import BatchedLU

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_order_one_is_a_division(dtype):
    g = torch.Generator().manual_seed(5)
    top = 1000 if dtype == torch.float64 else 120
    n = 4000
    mant = torch.rand((n, 5), generator=g, dtype=torch.float64) + 1.0
    ex = torch.randint(-2, 3, (n, 5), generator=g)
    ex[n // 2:] = torch.randint(-top, top, (n - n // 2, 5), generator=g)
    V = torch.ldexp(mant, ex) * (torch.randint(0, 2, (n, 5), generator=g) * 2 - 1)
    V[0, 1:] = torch.tensor([0.0, float("inf"), float("nan"), 1.0], dtype=torch.float64)
    V[1, 0], V[2, 0] = 2.0 ** -1060, float("inf")   # subnormal in FP64, zero in FP32
    V = V.to(dtype)
    V[3, 0] = 0.0                                    # a zero pivot: x / 0
    bl = BatchedLU([V[i:i + 1, :1] for i in range(n)], [V[i:i + 1, 1:] for i in range(n)], dtype=dtype)
    bl.restore()
    bl.run()
    torch.cuda.synchronize()
    X = bl.B.cpu().reshape(n, 4)
    torch.testing.assert_close(X, V[:, 1:] / V[:, :1], rtol=0, atol=0, equal_nan=True)
