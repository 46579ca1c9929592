"""A basis with an entry that is not finite (hef_orthonormalize, FP64): what the
mean-free column times R^-1 gives in FP64 arithmetic.  Its column's mean is not
finite, so every row of the output is NaN in all columns from the 64-column
block on that the column belongs to, and those columns are not kept; the blocks
before it are those of the finite columns (LAPACK's QR, tolerance of
test_gpu_ortho_f64.py)."""
import numpy as np
import pytest

from tests.test_gpu_ortho_f64 import EPS, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("K,c,row", [(12, 3, 100), (12, 0, 599), (64, 63, 0), (65, 64, 300),
                                     (150, 70, 17), (150, 149, 599), (150, 20, 5), (200, 128, 480)])
def test_nan_from_the_block_on(K, c, row, value):
    V = np.random.default_rng(K + c).standard_normal((600, K))
    good = 64 * (c // 64)
    V[row, c] = value
    Q, _, rank = run(V)
    assert np.isnan(Q[:, good:]).all()
    assert rank == good
    if good:
        A = V[:, :good] - V[:, :good].mean(0)
        Qr, Rr = np.linalg.qr(A)
        assert np.abs(Q[:, :good] - Qr * np.sign(np.diag(Rr))).max() <= (
            8 * (K + 8) * EPS * np.linalg.cond(A))


def test_overflowing_mean():
    # finite entries whose sum is not
    V = np.random.default_rng(1).standard_normal((500, 70))
    V[:, 66] = 1e308
    Q, _, rank = run(V)
    assert np.isfinite(Q[:, :64]).all() and np.isnan(Q[:, 64:]).all() and rank == 64
