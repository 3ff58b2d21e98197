"""Dense sampling where device memory is short: a full pattern's values T(z_j) are twice the size of the complex64
factor, so a slot that kept them would not fit where the factor does.  The residuals then form T from its
terms.

Bars: backward error 1e-14 after refinement, recomputed on the host to 1e-13."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


def full_nep(rs, n, seed=3):
    rng = np.random.default_rng([n, seed])
    A = rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n))
    cols = np.tile(np.arange(n, dtype=np.int32), n)
    vals = np.zeros((2, n * n), dtype=complex)
    vals[0] = A.ravel()
    vals[1, :: n + 1] = -1.0
    U = rng.normal(size=(n, 2)) + 1j * rng.normal(size=(n, 2))
    return A, U, rs.Nep(n, np.arange(n + 1, dtype=np.int64) * n, cols, vals, [(rs.F_CONST, []), (rs.F_Z, [])],
                        rs.RSRR_DENSE_LU)


def test_full_pattern_with_little_memory(rs):
    import torch
    _, U, small = full_nep(rs, 130)
    with small as h:
        h.sample(0.5, 0.3, 0.2, 2, 2, U, rs.RSRR_C64_IR, 1e-14, 20)
    n = 3000
    A, U, big = full_nep(rs, n)
    with big as h:
        # 0.8 of 256 MB are one slot's budget: 81 MB without T's values, 225 MB with them
        free = torch.cuda.mem_get_info()[0]
        ballast = torch.empty(free - (256 << 20), dtype=torch.uint8, device="cuda")
        try:
            h.sample(0.5, 0.3, 0.2, 2, 2, U, rs.RSRR_C64_IR, 1e-14, 20)
        finally:
            del ballast
            torch.cuda.empty_cache()
        X, eta = h.samples(), h.eta()
        assert h.info()["dense_lu"] == 1
    assert eta.max() <= 1e-14
    t = 2 * np.pi * (np.arange(2) + 0.5) / 2
    for j, z in enumerate(0.5 + 0.3 * np.cos(t) + 0.2j * np.sin(t)):
        Xj = X[:, 2 * j:2 * j + 2]
        r = U - (A @ Xj - z * Xj)
        assert np.all(np.linalg.norm(r, axis=0) <= 1e-13 * (np.linalg.norm(A, 1) * np.linalg.norm(Xj, axis=0) + np.linalg.norm(U, axis=0)))
