"""Products that user code asks for inside a callback of rsrr_solve (rsrr_zgemm, path 2, on another stream)
finish before they return, as they do outside of one; and a step that fails after a product of the same call gave
up is reported as the timeout it follows from."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


def test_product_in_a_callback_has_finished(rs):
    import torch
    m = 1500
    gen = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn(m, m, dtype=torch.complex128, device="cuda", generator=gen)
    B = torch.randn(m, m, dtype=torch.complex128, device="cuda", generator=gen)
    side = torch.cuda.Stream()
    seen, armed = [], [False]

    def f(z):
        if armed[0]:
            armed[0] = False
            C = torch.zeros(m, m, dtype=torch.complex128, device="cuda")
            torch.cuda.synchronize()
            rs.zgemm(2, A, B, C, M=m, N=m, K=m, lds=(m, m, m), stream=side.cuda_stream)
            seen.append((side.query(), C))
        return z

    n, N, L = 40, 8, 4
    rng = np.random.default_rng(3)
    d = np.concatenate([np.linspace(-0.8, 0.7, 6), 1.6 + 0.05 * np.arange(n - 6)])
    U = rng.normal(size=(n, L)) + 1j * rng.normal(size=(n, L))
    vals = np.stack([d, -np.ones(n)])
    fns = [(rs.F_CONST, []), rs.callback_fn(f, lambda z: 1.0)]
    with rs.Nep(n, np.arange(n + 1), np.arange(n), vals, fns) as h:
        h.sample(0.0, 1.2, 1.2, N, L, U, rs.RSRR_FP64, 1e-10)
        h.project(1e-14)
        armed[0] = True
        lam, _, _ = h.solve(100, 2, 1e3, 40, False)
    finished, C = seen[0]
    assert finished
    ref = B @ A  # the buffers are column-major there: C^T = B^T A^T
    assert torch.linalg.norm(C - ref) <= 1e-13 * torch.linalg.norm(ref)
    assert lam.size == 6


@pytest.mark.parametrize("kind,name", [(4, "ETIMEOUT"), (5, "ESINGULAR")])
def test_status_after_a_product_that_gave_up(rs, kind, name):
    with pytest.raises(rs.RsrrError) as e:
        rs.rsrr_selftest_bounded_wait(kind)
    assert e.value.name == name
