"""P = S^H (A S) of a stencil matrix on a smooth basis: A S is formed to its own rounding, not to that of
|A| |S|, which is a million times as large here.

Bar, derived from the product alone: |P - S^H A S|_ij <= n^(1/2) u |s_i| |A s_j| with a factor 4 for the GEMM's
complex terms, A s_j in extended precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


@pytest.mark.parametrize("phase", [1.0, 0.6 + 0.8j])
def test_stencil_on_smooth_basis(rs, phase):
    n, N, L = 1000, 12, 4
    h2 = (n + 1.0) ** 2
    rows = np.concatenate([np.arange(n), np.arange(n - 1), np.arange(1, n)])
    cols = np.concatenate([np.arange(n), np.arange(1, n), np.arange(n - 1)])
    a = np.concatenate([np.full(n, 2.0 * h2 / 3.0), np.full(2 * (n - 1), -h2 / 3.0)])
    order = np.lexsort((cols, rows))
    rows, cols, a = rows[order], cols[order], a[order] * phase
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))])
    x = np.arange(1, n + 1) / (n + 1)
    U = np.stack([np.sin(np.pi * (k + 1) * x) + np.sin(np.pi * (k + 5) * x) for k in range(L)], axis=1).astype(complex)
    vals = np.stack([a.astype(complex), -(rows == cols).astype(complex)])
    with rs.Nep(n, rowptr, cols, vals, [(rs.F_CONST, []), (rs.F_Z, [])]) as h:
        h.sample(100.0 * phase, 90.0, 90.0, N, L, U, rs.RSRR_FP64, 1e-10)
        h.project(1e-10)
        S, P = h.basis(), h.projected()[0]
    Sl = S.astype(np.clongdouble)
    AS = np.zeros_like(Sl)
    al = a.astype(np.clongdouble)
    np.add.at(AS, rows, al[:, None] * Sl[cols])
    ref = (Sl.conj().T @ AS).astype(complex)
    u = 2.0 ** -53
    norms = np.linalg.norm(AS.astype(complex), axis=0)
    assert np.all(np.abs(P - ref) <= 4 * np.sqrt(n) * u * norms[None, :])
