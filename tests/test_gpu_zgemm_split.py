"""The FP64 ZGEMM's tiles and K slices: tile edges (16 x 16 and the thin 64 x 4), every slice count
of a cluster (1, 2, 4, 8) with ragged slices, all operand forms, and the same bits on every run.

Bar: the rounding bound of a dot product of K complex terms summed in any order,
4 (K + 2) 2^-53 max |Re|, |Im| of a row times that of a column, plus beta C's rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


@pytest.mark.parametrize("M,N,K", [(16, 16, 31), (17, 15, 32), (15, 17, 65), (33, 9, 129), (64, 4, 127), (65, 5, 256),
                                   (200, 8, 300), (3, 1, 1000), (32, 233, 257), (700, 700, 16)])
@pytest.mark.parametrize("oa,ob", [(0, 0), (1, 2), (2, 1)])
def test_fp64_path_matches_reference(rs, M, N, K, oa, ob):
    import torch
    rng = np.random.default_rng([M, N, K, oa, ob])
    mk = lambda r, c: rng.normal(size=(r, c)) + 1j * rng.normal(size=(r, c))  # noqa: E731
    a, b, C0 = mk(M, K), mk(K, N), mk(M, N)
    st = lambda x, o: x if o == 0 else x.T if o == 1 else x.conj().T  # noqa: E731  (stored so that op(X) = x)
    dA, dB = (torch.from_numpy(np.ascontiguousarray(st(x, o).T)).cuda() for x, o in ((a, oa), (b, ob)))
    out = []
    for _ in range(2):
        dC = torch.from_numpy(np.ascontiguousarray(C0.T)).cuda()
        rs.zgemm(1, dA, dB, dC, oa, ob, 0.5 - 2j, 1.5 + 0.25j, M=M, N=N, K=K, lds=(dA.shape[1], dB.shape[1], M))
        torch.cuda.synchronize()
        out.append(dC.cpu().numpy().T)
    assert np.array_equal(out[0], out[1])
    ref = (0.5 - 2j) * (a @ b) + (1.5 + 0.25j) * C0
    inf = lambda x, ax: np.maximum(np.abs(x.real), np.abs(x.imag)).max(axis=ax)  # noqa: E731
    bound = 4 * (K + 2) * 2.0 ** -53 * 2.1 * 2 * np.outer(inf(a, 1), inf(b, 0)) + 2.0 ** -51 * np.abs(C0)
    assert np.all(np.abs(out[0] - ref) <= bound)
