"""The backward solve of the tensor-core band path gives a thread block 4, 8 or 16 right-hand sides,
by the number of points and columns of a batch: the shares of a chunk, the window and the partial
sums differ with it.  80 points keep every column of a point in one block (3, 7 and 14 columns: the
three forms, ragged); 20 columns take two blocks of 10; 6 points spread 18 columns over five blocks.

A0 has rows of modulus sum below 130 off the diagonal and 200 on it, so cond(T) < 6 and a solution
with backward error 2e-15 is within 1.2e-14 of the exact one; the bound leaves three digits for norms."""
import numpy as np
import pytest

import oracle
from gpu_util import rel_err_cols
from test_gpu_band_tc import banded_problem, rs, run  # noqa: F401  (rs is the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L", [(80, 1), (80, 3), (80, 7), (80, 14), (80, 20), (6, 18)])
def test_backward_solve_column_groups(rs, N, L):  # noqa: F811
    prob = banded_problem(450, 40, 37, seed=N + L, N=N, L=L, shift=200.0)
    X, eta, info = run(rs, prob, rs.RSRR_C64_IR | rs.RSRR_REFINE_FULL, 1e-10)
    assert info["band_lu_tc"] == 1 and info["dense_lu"] == 0
    ref, infos, _ = oracle.sample(prob)
    assert np.all(infos == 0)
    assert eta.max() <= 2e-15
    assert rel_err_cols(X, ref).max() < 1e-11


@pytest.mark.parametrize("N,L,kl,ku", [(6, 7, 40, 37), (40, 5, 12, 15), (60, 17, 3, 1), (80, 4, 40, 37)])
@pytest.mark.parametrize("fp64", [True, False])
def test_cuda_core_solves_column_split(rs, N, L, kl, ku, fp64):  # noqa: F811
    """The CUDA-core solves spread a point's columns over as many blocks as fill the device: one
    column each, uneven shares, more columns than a block has warps, and one block.  FP64 has no
    refinement: a backward error of a few (kl + ku + 2) u, below 1e-13, times cond < 6 stays below
    1e-11 too."""
    prob = banded_problem(450, kl, ku, seed=N + L, N=N, L=L, shift=200.0)
    if fp64:
        X, eta, info = run(rs, prob, rs.RSRR_FP64, 1e-10)
    else:
        X, eta, info = run(rs, prob, rs.RSRR_C64_IR | rs.RSRR_REFINE_FULL, 1e-10, flags=rs.RSRR_BAND_CUDA_CORES)
    assert info["band_lu_tc"] == 0 and info["dense_lu"] == 0
    ref, infos, _ = oracle.sample(prob)
    assert np.all(infos == 0)
    assert eta.max() <= 1e-13
    assert rel_err_cols(X, ref).max() < 1e-11


@pytest.mark.parametrize("N", [6, 45, 60])
@pytest.mark.parametrize("fp64,kl,ku", [(True, 70, 70), (True, 90, 5), (True, 3, 40), (False, 70, 70), (False, 5, 90)])
def test_cuda_core_factor_cluster_sizes(rs, N, fp64, kl, ku):  # noqa: F811
    """The CUDA-core factorisation gives a point a cluster of 4, 3 or 2 blocks by the number of points,
    and fewer where the band has few trailing columns.  The shifted band is diagonally dominant
    (row sums off the diagonal below 240, 330 on it): cond < 7, bounds as above."""
    prob = banded_problem(601, kl, ku, seed=N + kl, N=N, L=3, shift=330.0)
    if fp64:
        X, eta, info = run(rs, prob, rs.RSRR_FP64, 1e-10)
    else:
        X, eta, info = run(rs, prob, rs.RSRR_C64_IR | rs.RSRR_REFINE_FULL, 1e-10, flags=rs.RSRR_BAND_CUDA_CORES)
    assert info["band_lu_tc"] == 0 and info["dense_lu"] == 0
    ref, infos, _ = oracle.sample(prob)
    assert np.all(infos == 0)
    assert eta.max() <= 1e-13
    assert rel_err_cols(X, ref).max() < 1e-11


def test_cuda_core_factor_cluster_pivoting(rs):  # noqa: F811
    """Rows move at nearly every column (no shift) under a cluster of four blocks: the solutions'
    backward error.  The entries of L are at most 1 and those of U grow at most by some tens here, so eta stays below
    100 (kl + ku + 2) u = 3e-12."""
    prob = banded_problem(601, 60, 50, seed=5, N=6, L=3)
    X, eta, info = run(rs, prob, rs.RSRR_FP64, 1e-10)
    assert info["band_lu_tc"] == 0 and info["dense_lu"] == 0
    assert eta.max() <= 3e-12
