"""A wait that gives up while the last, smaller group of right-hand sides is refined ends the call with its status."""
import ctypes
import threading
import time

import pytest
import torch

from paper_1511_07174_gb300 import _lib, api, inputs

pytestmark = pytest.mark.gpu


def test_timeout_in_a_group_smaller_than_the_layout():
    # columns 0 .. 3 (zero) are done at once; column 4 is a group of its own in a layout of four,
    # with a tolerance it cannot reach: it is being refined when the limit drops to zero
    n, k = 200, 5
    A = inputs.uniform(n, 1, "cuda")
    A.diagonal().add_(n ** 0.5)
    B = torch.zeros((n, k), dtype=torch.float64, device="cuda")
    B[:, 4] = inputs.normal((n,), 2, "cuda")
    F, ipiv, _ = api.lu_factor_mixed(A, "bf16")
    Ac, Bc = api.colmajor(A), api.colmajor(B)
    X = api.colmajor(torch.zeros_like(B))
    lib = _lib.load()
    ws = torch.empty(lib.gbla_gmresir_workspace_nrhs(n, k, 50), dtype=torch.uint8, device="cuda")
    opts = _lib.GmresirOpts(0.0, 1e-8, 20000, 50, 1)
    st = (_lib.GmresirStats * k)()
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    old = api.get_wait_timeout_ns()
    rc = []
    call = threading.Thread(target=lambda: rc.append(lib.gbla_gmresir_solve_nrhs(
        n, k, p(Ac), n, p(F), n, p(ipiv), p(Bc), n, p(X), n, ctypes.byref(opts), st, p(ws), ws.numel(), stream)))
    try:
        call.start()
        time.sleep(0.3)
        api.set_wait_timeout_ns(0)
        call.join()
    finally:
        api.set_wait_timeout_ns(old)
    torch.cuda.synchronize()
    assert all(s.converged and s.outer == 0 for s in st[:4])
    assert rc == [1005]  # GBLA_ERR_TIMEOUT
    assert not st[4].converged and st[4].outer < 20000
