"""FP64 orthonormalisation (hef_orthonormalize) at the edges of its tensor-core
tiles, against LAPACK's QR.

Tolerances: CholQR2 and Householder QR both return the orthonormal factor to
c K eps cond(V) with a small constant; 8 (K + 8) eps cond(V) bounds their
difference, and 8 (K + 8) eps the orthogonality and (relative to the largest
entry of V's column) the residual V - 1 mu^T - Q R."""
import numpy as np
import pytest
import torch

from tests._gpu import DEV

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


def run(V):
    import paper_2511_06600_gb300 as hef
    n, K = V.shape
    d = torch.zeros(n, hef.padded_ld(K, torch.float64), dtype=torch.float64, device=DEV)
    d[:, :K] = torch.from_numpy(V).to(DEV)
    Q, R, rank = hef.orthonormalize(d, K, want_R=True)
    return Q[:, :K].cpu().numpy(), R.cpu().numpy(), int(rank)


def check(V, scale=None):
    n, K = V.shape
    Q, R, rank = run(V if scale is None else V * scale)
    A = V - V.mean(0)
    Qr, Rr = np.linalg.qr(A)
    s = np.sign(np.diag(Rr))
    s[s == 0] = 1
    tol = 8 * (K + 8) * EPS
    assert rank == K
    assert np.abs(Q.T @ Q - np.eye(K)).max() <= tol
    assert np.abs(Q.sum(0)).max() <= tol * np.sqrt(n)
    assert np.abs(Q - Qr * s).max() <= tol * np.linalg.cond(A)
    assert (np.tril(R, -1) == 0).all() and (np.diag(R) > 0).all()
    if scale is None:
        assert (np.abs(A - Q @ R).max(0) <= tol * np.abs(V).max(0) * np.sqrt(K)).all()


@pytest.mark.parametrize("n,K", [
    (65, 1), (64, 7), (129, 15), (127, 16), (513, 17), (1000, 48), (512, 63), (511, 64),
    (1537, 65), (1024, 127), (900, 128), (1100, 129), (4097, 160), (2000, 191), (1600, 257),
    (2100, 384), (2048, 511), (2304, 512), (90001, 20), (33000, 130)])
def test_against_lapack(n, K):
    check(np.random.default_rng(n + K).standard_normal((n, K)))


def test_column_scales_far_apart():
    # each column on its own scale, a spread that no common scale could hold
    rng = np.random.default_rng(1)
    check(rng.standard_normal((3000, 70)), 10.0 ** rng.integers(-120, 120, size=70))


def test_peaked_columns():
    # entries down to 2^-40 of their column's largest: the digits below the
    # peak's last one are rounded, which must stay at the level of eps times
    # the column's norm
    rng = np.random.default_rng(2)
    V = rng.standard_normal((5000, 33)) * 2.0 ** rng.integers(-40, 1, size=(5000, 1))
    check(V)


def test_zero_and_dependent_columns():
    rng = np.random.default_rng(3)
    V = rng.standard_normal((700, 20))
    V[:, 5] = 0.0
    V[:, 9] = V[:, 2] - 2 * V[:, 4]
    V[:, 13] = 3.25  # the constant: nothing left without its mean
    Q, R, rank = run(V)
    assert rank == 17
    for c in (5, 9, 13):
        assert (Q[:, c] == 0).all()
    keep = [c for c in range(20) if c not in (5, 9, 13)]
    assert np.abs(Q[:, keep].T @ Q[:, keep] - np.eye(17)).max() <= 8 * 28 * EPS


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_entry_that_is_not_finite(value):
    # its column is dropped and its row is lost; the other rows are those of
    # the basis without that column (zero weights of a dropped column)
    rng = np.random.default_rng(4)
    V = rng.standard_normal((600, 12))
    V[100, 3] = value
    Q, R, rank = run(V)
    assert np.isnan(Q[100]).all()
    assert rank < 12


def test_repeatable_and_independent_of_the_stream():
    rng = np.random.default_rng(5)
    V = rng.standard_normal((20011, 90))
    a = run(V)
    with torch.cuda.stream(torch.cuda.Stream()):
        b = run(V)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("dtype,K", [(torch.float64, 47), (torch.float64, 48), (torch.float64, 63),
                                     (torch.float64, 150), (torch.float64, 400),
                                     (torch.float32, 161), (torch.float32, 200),
                                     (torch.float32, 384), (torch.float32, 511)])
def test_elimination_over_the_grid(dtype, K):
    # K around the sizes at which the elimination moves to the grid, partial
    # panels, and dependent columns whose pivots must be dropped; the rank and
    # the orthogonality to 8 (K + 8) eps (FP32: the second pass leaves rounding
    # of the FP32 basis and of its tensor-core sums, 64 K eps)
    import paper_2511_06600_gb300 as hef
    rng = np.random.default_rng(K)
    n = 6 * K + 11
    V = rng.standard_normal((n, K))
    V[:, K // 2] = V[:, 1] + V[:, 3]
    V[:, K - 1] = 0
    d = torch.zeros(n, hef.padded_ld(K, dtype), dtype=dtype, device=DEV)
    d[:, :K] = torch.from_numpy(V).to(DEV)
    Q, R, rank = hef.orthonormalize(d, K, want_R=True)
    Q = Q[:, :K].double().cpu().numpy()
    assert int(rank) == K - 2
    assert (Q[:, K // 2] == 0).all() and (Q[:, K - 1] == 0).all()
    keep = [c for c in range(K) if c not in (K // 2, K - 1)]
    tol = 8 * (K + 8) * EPS if dtype == torch.float64 else 64 * K * np.finfo(np.float32).eps
    assert np.abs(Q[:, keep].T @ Q[:, keep] - np.eye(K - 2)).max() <= tol
    A = V - V.mean(0)
    res = np.abs(A - Q @ R.cpu().numpy()).max(0)
    assert (res[keep] <= tol * np.abs(V).max() * np.sqrt(K)).all()
