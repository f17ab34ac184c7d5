"""The FP64 trailing update as digit products on the tensor cores (LU with nb a
multiple of 128, Cholesky with scratch) against the CPU oracle.

Tolerances as in the FP64 LU tests: identical pivots (asserted only where the
oracle's smallest pivot gap allows), factors within 1e-11 of the largest entry,
dyadic products bit for bit (their digits and sums are exact). Operands that
the digits represent badly -- rows graded over many magnitudes, magnitudes
beyond 2^+-450, infinities -- must take the FP64 path tile by tile: compared
row by row, relative to each row's own scale, which a loss of the small
elements' digits would miss by many orders of magnitude.
"""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_1511_07174_gb300 import _lib, api, inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _lu(A, nb):
    LU, ipiv, info = api.lu_factor(A.to(DEV), nb=nb)
    torch.cuda.synchronize()
    return LU.cpu().numpy(), ipiv.cpu().numpy(), int(info.item())


# one element, one row / column short of and past a 128-tile, several tiles, ragged K
@pytest.mark.parametrize("n,nb", [(129, 128), (255, 128), (256, 128), (257, 128), (385, 256), (511, 256),
                                  (513, 256), (641, 128), (900, 256), (1300, 256)])
def test_lu_digits_match_oracle(n, nb):
    A = inputs.uniform(n, seed=40 + n)
    An = np.asfortranarray(A.numpy())
    assert oracle.min_pivot_gap(An) > 1e-10
    LUo, ipo, info_o = oracle.getrf(An)
    LUg, ipg, info_g = _lu(A, nb)
    assert info_g == info_o == 0
    assert np.array_equal(ipg, ipo)
    assert np.abs(LUg - LUo).max() <= 1e-11 * max(1.0, np.abs(LUo).max())


@pytest.mark.parametrize("n,nb", [(300, 128), (777, 256)])
def test_lu_digits_dyadic_exact(n, nb):
    A, L0, U0, perm = inputs.dyadic_lu(n, seed=70 + n)
    LUg, ipg, info = _lu(A, nb)
    L, U = oracle.unpack_lu(LUg)
    assert info == 0
    assert np.array_equal(L, L0.numpy()) and np.array_equal(U, U0.numpy())


def _by_rows(LUg, LUo, tol):
    n = LUo.shape[0]
    for g, o in ((np.triu(LUg), np.triu(LUo)), (np.tril(LUg, -1), np.tril(LUo, -1))):
        scale = np.abs(o).max(axis=1)
        d = np.abs(g - o).max(axis=1)
        assert np.all(d <= tol * scale + 0.0), float((d / np.maximum(scale, 1e-300)).max())
    assert n > 0


@pytest.mark.parametrize("decades", [6, 12])
def test_lu_graded_rows_keep_their_digits(decades):
    n = 520
    A = inputs.uniform(n, seed=3)
    g = torch.Generator().manual_seed(4)
    A = A * torch.pow(10.0, -decades * torch.rand((n, 1), generator=g, dtype=torch.float64))
    An = np.asfortranarray(A.numpy())
    assert oracle.min_pivot_gap(An) > 1e-10
    LUo, ipo, _ = oracle.getrf(An)
    LUg, ipg, info = _lu(A, 128)
    assert info == 0 and np.array_equal(ipg, ipo)
    _by_rows(LUg, LUo, 1e-9)


@pytest.mark.parametrize("scale", [2.0 ** -700, 2.0 ** 700, 2.0 ** -1000])
def test_lu_extreme_magnitudes(scale):
    """Powers of two move the exponents only: the same factors, scaled."""
    n = 400
    A = inputs.uniform(n, seed=8)
    LU1, ip1, _ = _lu(A, 128)
    LUs, ips, info = _lu(A * scale, 128)
    assert info == 0 and np.array_equal(ip1, ips)
    LUo, _, _ = oracle.getrf(np.asfortranarray(A.numpy()))
    assert np.abs(np.triu(LUs) / scale - np.triu(LUo)).max() <= 1e-11 * np.abs(LUo).max()
    assert np.abs(np.tril(LUs, -1) - np.tril(LUo, -1)).max() <= 1e-11


def test_lu_infinity_stays_in_its_column():
    """An infinity to the right of the first block reaches only its own column."""
    n = 400
    A = inputs.uniform(n, seed=9)
    LU1, ip1, _ = _lu(A, 128)
    A2 = A.clone()
    A2[0, n - 1] = float("inf")
    LU2, ip2, _ = _lu(A2, 128)
    assert np.abs(LU2[:, :n - 1] - LU1[:, :n - 1]).max() <= 1e-11 * np.abs(LU1).max()
    assert not np.isfinite(LU2[:, n - 1]).all()


def test_lu_small_workspace_takes_the_fp64_pipe():
    """The workspace size of before is accepted; both paths give the oracle's factors."""
    n, nb = 600, 256
    L = _lib.load()
    small, large = L.gbla_lu_factor_workspace(n, nb), L.gbla_lu_factor_workspace_tensor(n, nb)
    assert small < large
    A = inputs.uniform(n, seed=12)
    LUo, ipo, _ = oracle.getrf(np.asfortranarray(A.numpy()))
    LU = api.colmajor(A.to(DEV), torch.float64, copy=True)
    ipiv = torch.empty(n, dtype=torch.int32, device=DEV)
    info = torch.zeros(1, dtype=torch.int32, device=DEV)
    ws = torch.empty(small, dtype=torch.uint8, device=DEV)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    assert L.gbla_lu_factor(n, p(LU), n, p(ipiv), p(info), nb, p(ws), small,
                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert np.array_equal(ipiv.cpu().numpy(), ipo)
    assert np.abs(LU.cpu().numpy() - LUo).max() <= 1e-11 * np.abs(LUo).max()


@pytest.mark.parametrize("n,nb", [(65, 64), (200, 64), (257, 128), (700, 256), (1000, 0), (1100, 192)])
def test_chol_digits_match_oracle(n, nb):
    S = inputs.spd(n, seed=n)
    F, info = api.chol_factor(S.to(DEV), nb=nb)
    torch.cuda.synchronize()
    Lo, info_o = oracle.potrf(np.asfortranarray(S.numpy()))
    assert int(info.item()) == info_o == 0
    Fg = F.cpu().numpy()
    assert np.abs(np.tril(Fg) - np.tril(Lo)).max() <= 1e-12 * np.abs(np.tril(Lo)).max()
    assert np.array_equal(np.triu(Fg, 1), np.triu(S.numpy(), 1))


def test_chol_without_scratch_agrees():
    n = 500
    S = inputs.spd(n, seed=2)
    F1, _ = api.chol_factor(S.to(DEV), nb=128)
    F2 = api.colmajor(S.to(DEV), torch.float64, copy=True)
    info = torch.zeros(1, dtype=torch.int32, device=DEV)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    assert _lib.load().gbla_chol_factor(n, p(F2), n, p(info), 128,
                                        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    assert float((F1 - F2).abs().max()) <= 1e-13 * float(F1.abs().max())


def test_digit_update_gives_up_cleanly():
    """Wait limit 0: every wait of the update's mbarriers gives up, the call ends
    with the status, the context stays usable and the next call is right."""
    A = inputs.uniform(1024, seed=9).to(DEV)
    S = inputs.spd(600, seed=1).to(DEV)
    old = api.get_wait_timeout_ns()
    try:
        api.set_wait_timeout_ns(0)
        _, ipiv, info = api.lu_factor(A, nb=128)
        _, info_c = api.chol_factor(S, nb=128)
        torch.cuda.synchronize()
        assert int(info.item()) == -1000 and int(info_c.item()) == -1000
    finally:
        api.set_wait_timeout_ns(old)
    test_lu_digits_match_oracle(641, 128)
