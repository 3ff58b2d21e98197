"""The basis S of rsrr_project for probing matrices of any size.  Below 1e-77 the squared inner products of
the Jacobi's columns underflow and the sweeps end early; S must still be orthonormal and span the samples.

Bars: as in the projection's other tests, |S^H S - I| < 1e-12 and |X - S S^H X|_2 <= 20 delta sigma_1 +
1e-15 |X|_F, X scaled back."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


@pytest.mark.parametrize("scale", [1e60, 1.0, 1e-70, 1e-77, 1e-78, 1e-79, 1e-80])
def test_orthonormal_at_any_scale(rs, scale):
    n, N, L = 60, 6, 8
    rng = np.random.default_rng(0)
    d = np.linspace(1.0, 2.0, n)
    U = scale * (rng.normal(size=(n, L)) + 1j * rng.normal(size=(n, L)))
    vals = np.stack([d, -np.ones(n)])
    with rs.Nep(n, np.arange(n + 1), np.arange(n), vals, [(rs.F_CONST, []), (rs.F_Z, [])]) as h:
        h.sample(1.5, 0.9, 0.9, N, L, U, rs.RSRR_FP64, 1e-10)
        h.project(1e-14)
        X, S = h.samples() / scale, h.basis()
    assert np.linalg.norm(S.conj().T @ S - np.eye(S.shape[1])) < 1e-12
    assert np.linalg.norm(X - S @ (S.conj().T @ X), 2) <= 20e-14 * np.linalg.norm(X, 2) + 1e-15 * np.linalg.norm(X)
