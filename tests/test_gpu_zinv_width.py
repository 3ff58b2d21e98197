"""The block width of the batched inverse changes where a panel of k rows no longer fits shared memory
(32 columns up to k = 450, 16 up to 900, 8 beyond), and the triangular inverses take the panel's
place: sizes on both sides of each line, the largest with 8 columns, and last panels of one column.
Bounds as for the other sizes (normwise residual and difference at FP64 rounding level)."""
import numpy as np
import pytest

from test_gpu_zinv import check, rand, rs, run  # noqa: F401  (rs is the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", [1, 2])
@pytest.mark.parametrize("k", [385, 404, 449, 450, 451, 900, 901])
def test_inverse_block_widths(rs, path, k):  # noqa: F811
    rng = np.random.default_rng([k, path])
    mats = [rand(rng, k) for _ in range(2)]
    X, info = run(rs, mats, path)
    assert np.all(info == 0)
    for A, Xi in zip(mats, X):
        check(A, Xi)
