"""The reduced eigenproblem's size range through whole passes: diagonal NEPs with a known number of
eigenvalues inside the contour, from one (no rotation at all) over 31, 33 and 81 (one more than the
kernel keeps in shared memory) to a conjugate-pair spectrum whose Wilkinson shifts are complex.

Bar: eigenvalues to 1e-9 of their closed form, as everywhere in the pipeline tests."""
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


@pytest.mark.parametrize("inside", [1, 2, 3, 31, 33, 80, 81])
@pytest.mark.parametrize("complex_pairs", [False, True])
def test_eigenvalues_of_a_diagonal(rs, inside, complex_pairs):
    t = np.linspace(-0.9, 0.83, inside) if inside > 1 else np.array([0.3])
    d = t + (0.35j * (-1.0) ** np.arange(inside) if complex_pairs else 0)
    far = 3.0 + 0.2 * np.arange(40)
    d = np.concatenate([d * (0.9 if complex_pairs else 1.0), far]).astype(complex)
    n = d.size
    L = 8
    rng = np.random.default_rng([inside, complex_pairs])
    U = rng.normal(size=(n, L)) + 1j * rng.normal(size=(n, L))
    with rs.Nep(n, np.arange(n + 1), np.arange(n), np.stack([d, -np.ones(n)]), [(rs.F_CONST, []), (rs.F_Z, [])]) as h:
        h.sample(0.0, 1.2, 1.2, 32, L, U, rs.RSRR_FP64, 1e-10)
        h.project(1e-14)
        lam, V, res = h.solve(500, 2, 1e3, 200, True)
    assert lam.size == inside
    assert match(lam, d[:inside]) < 1e-9
