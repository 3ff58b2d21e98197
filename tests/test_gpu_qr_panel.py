"""The Householder QR's panel kernel through rsrr_project: sample matrices whose row counts fall on
and around the kernel's row groups of 32, panels that are not full, fewer rows than columns, columns that
are zero from some row on (identity reflectors), and enough rows that a CTA's share leaves shared memory.

Bars: S orthonormal to 1e-12 and |X - S S^H X|_2 <= 20 delta sigma_1 + 1e-15 |X|_F (the truncation level
and the QR's rounding), singular values above 1e-6 sigma_1 to 1e-9."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


def project_diagonal(rs, n, N, L, U):
    """Samples X_j = (D - z_j I)^{-1} U of a diagonal T on a circle, projected on the device."""
    d = np.linspace(1.0, 2.0, n)
    rp, ci = np.arange(n + 1), np.arange(n)
    vals = np.stack([d, -np.ones(n)]).astype(complex)
    with rs.Nep(n, rp, ci, vals, [(rs.F_CONST, []), (rs.F_Z, [])]) as h:
        h.sample(1.5, 0.9, 0.9, N, L, U, rs.RSRR_FP64, 1e-10)
        X = h.samples()
        h.project(1e-14)
        return X, h.basis(), h.sigma()


@pytest.mark.parametrize("n,N,L", [(1, 1, 1), (5, 3, 2), (31, 2, 16), (32, 4, 8), (33, 11, 3), (65, 1, 33), (97, 7, 5),
                                   (1000, 5, 13), (4863, 9, 4), (4865, 3, 11)])
def test_panels(rs, n, N, L):
    rng = np.random.default_rng([n, N, L])
    U = rng.normal(size=(n, L)) + 1j * rng.normal(size=(n, L))
    if L > 2:
        U[n // 2:, 1] = 0.0
        U[: n // 2, 2] = 0.0
    X, S, sig = project_diagonal(rs, n, N, L, U)
    ref = np.linalg.svd(X, compute_uv=False)
    assert np.linalg.norm(S.conj().T @ S - np.eye(S.shape[1])) < 1e-12
    assert np.linalg.norm(X - S @ (S.conj().T @ X), 2) <= 20e-14 * ref[0] + 1e-15 * np.linalg.norm(X)
    top = ref[ref > 1e-6 * ref[0]]
    assert np.allclose(sig[:top.size], top, rtol=1e-9, atol=0)


def test_rows_beyond_shared_memory(rs):
    n, N, L = 70001, 2, 20
    rng = np.random.default_rng(7)
    U = rng.normal(size=(n, L)) + 1j * rng.normal(size=(n, L))
    X, S, sig = project_diagonal(rs, n, N, L, U)
    assert np.linalg.norm(S.conj().T @ S - np.eye(S.shape[1])) < 1e-12
    assert np.linalg.norm(X - S @ (S.conj().T @ X)) <= 1e-13 * np.linalg.norm(X)
    ref = np.linalg.svd(np.linalg.qr(X, mode="r"), compute_uv=False)
    assert np.allclose(sig, ref, rtol=1e-9, atol=1e-13 * ref[0])
