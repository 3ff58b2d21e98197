"""Dense sampling beyond the sizes where panels have leaves of eight columns: leaves of four (n > 3088 in
complex64, n > 1560 in FP64), panels in global memory (n > 6176, n > 3120), both on clusters, with fewer
right-hand sides than a cluster has CTAs.

Bars: backward error 1e-13 in FP64 and 1e-14 after refinement, as in the other dense tests, and ten times that
recomputed on the host."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


@pytest.mark.parametrize("n,L,prec", [(3089, 1, "c64"), (3150, 3, "c64"), (6200, 1, "c64"), (1561, 1, "fp64"),
                                      (1700, 5, "fp64"), (3130, 2, "fp64")])
def test_dense_points(rs, n, L, prec):
    rng = np.random.default_rng([n, L])
    # a random sparse pattern without its diagonal: every step of the LU pivots
    rows = np.repeat(np.arange(n), 6)
    cols = (rows + rng.integers(1, n, size=rows.size)) % n
    v = rng.normal(size=rows.size) + 1j * rng.normal(size=rows.size)
    A = sp.csr_matrix((v, (rows, cols)), shape=(n, n)) + sp.csr_matrix(np.roll(np.eye(n), 1, axis=1) * 4.0)
    T = (abs(A) + sp.identity(n)).tocsr()
    T.sort_indices()
    r = np.repeat(np.arange(n), np.diff(T.indptr))
    vals = np.stack([np.asarray(A[r, T.indices]).ravel(), -(r == T.indices).astype(complex)])
    U = rng.normal(size=(n, L)) + 1j * rng.normal(size=(n, L))
    fp64 = prec == "fp64"
    tol = 1e-13 if fp64 else 1e-14
    with rs.Nep(n, T.indptr, T.indices, vals, [(rs.F_CONST, []), (rs.F_Z, [])], rs.RSRR_DENSE_LU) as h:
        h.sample(0.5, 0.3, 0.2, 2, L, U, rs.RSRR_FP64 if fp64 else rs.RSRR_C64_IR, 1e-12 if fp64 else 1e-14, 20)
        X, eta = h.samples(), h.eta()
        assert h.info()["dense_lu"] == 1
    assert eta.max() <= tol
    t = 2 * np.pi * (np.arange(2) + 0.5) / 2
    for j, z in enumerate(0.5 + 0.3 * np.cos(t) + 0.2j * np.sin(t)):
        M = A - z * sp.identity(n)
        Xj = X[:, L * j:L * (j + 1)]
        bound = abs(M).sum(axis=0).max() * np.linalg.norm(Xj, axis=0) + np.linalg.norm(U, axis=0)
        assert np.all(np.linalg.norm(U - M @ Xj, axis=0) <= 10 * tol * bound)
