"""The one-sided Jacobi's rotation through rsrr_project on two unknowns: one FP64 rotation makes the pair of
columns orthogonal to rounding, so the second sweep finds nothing above the stopping level of 1e-10 and
is the last one, whatever the columns."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


@pytest.mark.parametrize("seed", range(6))
def test_one_rotation_settles_a_pair(rs, seed):
    rng = np.random.default_rng(seed)
    A = rng.normal(size=(2, 2)) + 1j * rng.normal(size=(2, 2))
    U = rng.normal(size=(2, 2)) + 1j * rng.normal(size=(2, 2))
    vals = np.stack([A.ravel(), -np.eye(2).ravel()])
    with rs.Nep(2, np.array([0, 2, 4]), np.array([0, 1, 0, 1]), vals, [(rs.F_CONST, []), (rs.F_Z, [])]) as h:
        h.sample(0.0, 4.0, 4.0, 4, 2, U, rs.RSRR_FP64, 1e-10)
        h.project(1e-14)
        ref = np.linalg.svd(h.samples(), compute_uv=False)
        assert h.info()["jacobi_sweeps_project"] == 2
        assert np.allclose(h.sigma(), ref, rtol=1e-14, atol=0)
