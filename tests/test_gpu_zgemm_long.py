"""Products of few outputs and long K on the FP64 cores: a tile's K range is cut over several clusters whose sums
are folded from a workspace.  Every tile shape (16 x 16, 64 x 4, 4 x 64), remainders of K, beta, batches and leading
dimensions above the sizes.

Bars: |C - ref|_ij <= 4 K^(1/2) u (|op(A)| |op(B)|)_ij + 2 u |beta C|, ref from torch's complex128 product, whose
own error the factor 4 includes.  For the times: the path chosen by shape takes at most 1.5 times the faster of the
two (both timed here), and the FP64 path at most four times what a product of as much work with as many
tiles as the device has SMs takes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1510_07522_gb300 as rs
    return rs


def operands(M, N, K, opA, opB, batch, pad=0):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(M + N + K)
    ra, ca = (M, K) if opA == 0 else (K, M)
    rb, cb = (K, N) if opB == 0 else (N, K)
    # row-major [batch][columns][ld] is column-major with leading dimension ld
    make = lambda r, c: torch.randn(batch, c, r + pad, dtype=torch.complex128, device="cuda", generator=gen)
    return make(ra, ca), make(rb, cb), make(M, N)


def op(X, rows, o):
    X = X[:, :, :rows].transpose(1, 2)
    return X if o == 0 else (X.transpose(1, 2) if o == 1 else X.transpose(1, 2).conj())


@pytest.mark.parametrize("M,N,K,opA,opB,batch", [(8, 8, 1023, 2, 0, 1), (8, 8, 1024, 0, 0, 1), (16, 16, 40000, 2, 0, 1),
                                                 (17, 9, 9999, 0, 2, 2), (2, 130, 5001, 2, 0, 1), (8, 64, 4097, 1, 0, 3),
                                                 (65, 5, 3000, 2, 1, 1), (100, 1, 70001, 0, 1, 1), (1, 1, 100003, 2, 0, 1),
                                                 (5, 300, 64, 0, 0, 1)])
def test_against_torch(rs, M, N, K, opA, opB, batch):
    import torch
    pad = 3
    A, B, C = operands(M, N, K, opA, opB, batch, pad)
    C0 = C.clone()
    alpha, beta = 0.7 - 0.2j, -0.4 + 0.9j
    rows = lambda o, r, c: r if o == 0 else c
    ra, rb = rows(opA, M, K), rows(opB, K, N)
    ld = lambda X: X.shape[2]
    rs.zgemm(1, A, B, C, opA, opB, alpha, beta, M=M, N=N, K=K, batch=batch, lds=(ld(A), ld(B), ld(C)),
             strides=(A[0].numel(), B[0].numel(), C[0].numel()))
    torch.cuda.synchronize()
    a, b = op(A, ra, opA), op(B, rb, opB)
    got, old = op(C, M, 0), op(C0, M, 0)
    ref = alpha * (a @ b) + beta * old
    u = 2.0 ** -53
    bound = 4 * np.sqrt(K) * u * abs(alpha) * (a.abs() @ b.abs()) + 2 * u * (beta * old).abs()
    assert bool(((got - ref).abs() <= bound).all())
    assert torch.equal(C[:, :, M:], C0[:, :, M:])


def time_us(rs, path, M, N, K, opA):
    import torch
    A, B, C = operands(M, N, K, opA, 0, 1)
    call = lambda: rs.zgemm(path, A, B, C, opA, 0, M=M, N=N, K=K, lds=(A.shape[2], K, M))
    for _ in range(3):
        call()
    a, b = torch.cuda.Event(True), torch.cuda.Event(True)
    torch.cuda.synchronize()
    a.record()
    for _ in range(5):
        call()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / 5 * 1e3


@pytest.mark.parametrize("M,N,K,opA", [(32, 8, 100000, 2), (600, 8, 100000, 2), (16, 3, 360000, 1), (2, 2048, 40000, 2),
                                       (5, 300, 100000, 2), (600, 8, 10000, 2), (40000, 4, 600, 0), (40000, 8, 233, 0)])
def test_shape_takes_the_faster_path(rs, M, N, K, opA):
    chosen, fp64, tc = (time_us(rs, p, M, N, K, opA) for p in (0, 1, 2))
    assert chosen <= 1.5 * min(fp64, tc), (chosen, fp64, tc)


@pytest.mark.parametrize("M,N,K", [(32, 8, 100000), (16, 16, 60000), (8, 8, 300000)])
def test_long_k_fills_the_device(rs, M, N, K):
    # the same work as 256 tiles of 16 x 16 (256 x 256 outputs)
    even = time_us(rs, 1, 256, 256, max(16, M * N * K // 65536), 2)
    assert time_us(rs, 1, M, N, K, 2) <= 4 * even + 20
