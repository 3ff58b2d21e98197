"""Dense LU panels by size class: whole panel in shared memory, leaves of 16, of 8 and of 4 columns (the
class follows from n and the precision), with panel tails of every kind and pivoting at every step.

Bars: backward error 1e-13 in FP64 and 1e-14 after refinement, as in the dense tests, and the
solution of numpy's LU to 1e-8."""
import numpy as np
import pytest

from gpu_util import rel_err_cols

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


@pytest.mark.parametrize("n,prec", [(63, "c64"), (65, "c64"), (385, "c64"), (388, "c64"), (1543, "c64"), (1610, "c64"),
                                    (129, "fp64"), (200, "fp64"), (773, "fp64"), (1549, "fp64")])
def test_dense_points(rs, n, prec):
    rng = np.random.default_rng([n, 3])
    A = rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n))
    A[np.arange(n), np.arange(n)] = 0.0           # every step pivots
    A[:, 0] *= 1e3
    rows, cols = np.divmod(np.arange(n * n), n)
    vals = np.zeros((2, n * n), dtype=complex)
    vals[0] = A.ravel()
    vals[1, rows == cols] = -1.0
    U = rng.normal(size=(n, 9)) + 1j * rng.normal(size=(n, 9))
    fp64 = prec == "fp64"
    with rs.Nep(n, np.arange(n + 1) * n, cols, vals, [(rs.F_CONST, []), (rs.F_Z, [])], rs.RSRR_DENSE_LU) as h:
        h.sample(0.5, 0.3, 0.2, 2, 9, U, rs.RSRR_FP64 if fp64 else rs.RSRR_C64_IR, 1e-12 if fp64 else 1e-14, 20)
        X, eta = h.samples(), h.eta()
        assert h.info()["dense_lu"] == 1
    assert eta.max() <= (1e-13 if fp64 else 1e-14)
    t = 2 * np.pi * (np.arange(2) + 0.5) / 2
    z = 0.5 + 0.3 * np.cos(t) + 0.2j * np.sin(t)
    ref = np.concatenate([np.linalg.solve(A - x * np.eye(n), U) for x in z], axis=1)
    assert rel_err_cols(X, ref).max() < 1e-8
