"""Cholesky of one diagonal block, which takes no scratch: the factors and the argument checks of the others."""
import ctypes

import pytest
import torch

from paper_1511_07174_gb300 import _lib, api, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 17, 63, 64, 65])
@pytest.mark.parametrize("nb", [0, 64, 256])
def test_same_as_with_scratch(n, nb):
    S = inputs.spd(n, seed=n).cuda()
    if n > 2:
        S[n - 1, n - 1] = -1.0  # stops in the last column
    F, info = api.chol_factor(S, nb=nb)
    L = _lib.load()
    G = api.colmajor(S, torch.float64, copy=True)
    gi = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(L.gbla_chol_factor_workspace(n, nb), dtype=torch.uint8, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert L.gbla_chol_factor_ws(n, p(G), n, p(gi), nb, p(ws), ws.numel(),
                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    assert torch.equal(F, G) and torch.equal(info, gi) and int(info.item()) == (n if n > 2 else 0)


@pytest.mark.parametrize("n", [0, 5, 64, 65])
@pytest.mark.parametrize("nb", [-64, 32, 96, 320])
def test_block_sizes_that_are_refused(n, nb):
    with pytest.raises(api.GblaError):
        api.chol_factor(inputs.spd(max(n, 1), seed=1).cuda()[:n, :n], nb=nb)
