"""gbla_lu_factor with the default block size accepts the scratch of 256-wide blocks."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_1511_07174_gb300 import _lib, api, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 700])
def test_scratch_of_wider_blocks(n):
    L = _lib.load()
    nbytes = L.gbla_lu_factor_workspace(n, 256)
    assert nbytes < L.gbla_lu_factor_workspace(n, 0)
    A = inputs.uniform(n, seed=12)
    LUo, ipo, _ = oracle.getrf(np.asfortranarray(A.numpy()))
    LU = api.colmajor(A.cuda(), torch.float64, copy=True)
    ipiv = torch.empty(n, dtype=torch.int32, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert L.gbla_lu_factor(n, p(LU), n, p(ipiv), p(info), 0, p(ws), nbytes, stream) == 0
    torch.cuda.synchronize()
    assert int(info.item()) == 0 and np.array_equal(ipiv.cpu().numpy(), ipo)
    assert np.abs(LU.cpu().numpy() - LUo).max() <= 1e-11 * np.abs(LUo).max()
    assert L.gbla_lu_factor(n, p(LU), n, p(ipiv), p(info), 0, p(ws), nbytes - 256, stream) == 1001
