"""Moments and traces of the reduced solve by their number of columns and terms (one, a full group of
four, five, eight, and nine, which goes to the GEMM), for a k below and above the moments kernel's range.

Bar: eigenvalues to 1e-9 of the closed form, the winding number to 1e-8 of the count."""
import numpy as np
import pytest

from gpu_util import match

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


@pytest.mark.parametrize("J,K,n,N,L", [(2, 1, 60, 16, 8), (5, 2, 60, 16, 8), (8, 4, 60, 16, 8), (9, 5, 60, 16, 8),
                                       (2, 2, 300, 30, 10), (5, 4, 300, 30, 10), (9, 5, 300, 30, 10)])
def test_terms_and_moments(rs, J, K, n, N, L):
    d = np.concatenate([np.linspace(-0.8, 0.7, 12), 1.6 + 0.02 * np.arange(n - 12)]).astype(complex)
    rng = np.random.default_rng([J, K, n])
    w = rng.uniform(0.5, 1.5, J - 1)
    vals = np.concatenate([np.outer(w / w.sum(), d), -np.ones((1, n))])   # the constant part in J - 1 terms
    fns = [(rs.F_CONST, [])] * (J - 1) + [(rs.F_Z, [])]
    U = rng.normal(size=(n, L)) + 1j * rng.normal(size=(n, L))
    with rs.Nep(n, np.arange(n + 1), np.arange(n), vals, fns) as h:
        h.sample(0.0, 1.2, 1.2, N, L, U, rs.RSRR_FP64, 1e-10)
        h.project(1e-14)
        lam, V, res = h.solve(400, K, 1e3, 200, True)
        info = h.info()
    assert abs(info["winding_re"] - 12) < 1e-8 and abs(info["winding_im"]) < 1e-8
    assert lam.size == 12 and match(lam, d[:12]) < 1e-9
