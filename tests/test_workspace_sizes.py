"""Scratch sizes: what serves an order serves every smaller one."""
import pytest

from paper_1511_07174_gb300 import _lib

SIZES = {
    "backward_error": lambda L, n: L.gbla_backward_error_workspace(n, 8),
    "gmresir": lambda L, n: L.gbla_gmresir_workspace(n, 1),
    "gmresir_nrhs": lambda L, n: L.gbla_gmresir_workspace_nrhs(n, 4, 2),
    "krylov": lambda L, n: L.gbla_krylov_workspace(n, 1),
    "lu_factor": lambda L, n: L.gbla_lu_factor_workspace(n, 0),
    "lu_factor_tensor": lambda L, n: L.gbla_lu_factor_workspace_tensor(n, 0),
    "lu_solve": lambda L, n: L.gbla_lu_solve_workspace(n, 5),
    "chol_factor": lambda L, n: L.gbla_chol_factor_workspace(n, 0),
    "chol_solve": lambda L, n: L.gbla_chol_solve_workspace(n, 5),
    "lu_factor_mixed": lambda L, n: L.gbla_lu_factor_mixed_workspace(n, 256, 6),
}


@pytest.mark.parametrize("name", sorted(SIZES))
def test_sizes_do_not_decrease(name):
    L = _lib.load()
    last = 0
    for n in range(0, 20001):
        size = SIZES[name](L, n)
        assert size >= last, n
        last = size
