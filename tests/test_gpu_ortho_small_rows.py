"""FP64 orthonormalisation (hef_orthonormalize) of bases with rows far below their
columns' largest entries: the differences of such rows to rounding of the rows'
own size, as FP64 arithmetic gives them, and with them the scores of hyperedges
whose pins all lie in such rows.

The bases are [X; -X], whose column means are zero, so that a small row stays
small; half the difference of a row and its mirror image is the row.  (A row by
itself carries the rounding of the column means, one shift for all rows, which
scores do not see.)  Reference: Gram-Schmidt done twice in numpy.longdouble (64 bits of
mantissa or more).  A row of Q has the error of the triangular factor, which
multiplies the row, and of its own multiply-adds, which are bounded by
eps |V_r| |R^-1| <= eps |Q_r| |R| |R^-1|: 8 (K + 8) eps cond(V) |Q_r| bounds both
(the constant of test_gpu_ortho_f64.py)."""
import numpy as np
import pytest
import torch

from tests._gpu import DEV, to_dev
from tests._hypergraphs import from_lists
from tests.test_gpu_ortho_f64 import EPS, run

pytestmark = pytest.mark.gpu


def reference(V):
    Q = V.astype(np.longdouble)
    for i in range(V.shape[1]):
        for _ in range(2):
            if i:
                Q[:, i] -= Q[:, :i] @ (Q[:, :i].T @ Q[:, i])
        Q[:, i] /= np.sqrt((Q[:, i] ** 2).sum())
    return Q


def check_rows(X):
    V = np.concatenate([X, -X])
    n, K = X.shape
    Q, _, rank = run(V)
    want = reference(V)
    assert rank == K
    half = (Q[:n].astype(np.longdouble) - Q[n:]) / 2
    err = np.abs(half - want[:n]).max(1)
    tol = 8 * (K + 8) * EPS * np.linalg.cond(V) * np.sqrt((want[:n] ** 2).sum(1))
    assert (err <= tol).all(), float((err / tol).max())
    return Q, want


@pytest.mark.parametrize("s", [10, 20, 30, 40, 60])
@pytest.mark.parametrize("K", [1, 12])
def test_one_small_row(K, s):
    X = np.random.default_rng(s).standard_normal((500, K))
    X[123] *= 2.0 ** -s
    check_rows(X)


@pytest.mark.parametrize("n,K", [(100, 12), (65, 20), (350, 64), (400, 70), (450, 130), (800, 200)])
def test_every_row_on_its_own_scale(n, K):
    # most outputs lie below the digits' line: several blocks of 64 columns,
    # the last of 1, 2 or 4 octets of columns, tiles of rows that end within one
    rng = np.random.default_rng(n + K)
    X = rng.standard_normal((n, K)) * 2.0 ** -rng.integers(0, 41, size=(n, 1))
    X[:2 * K] = rng.standard_normal((2 * K, K))[:n]
    check_rows(X)


@pytest.mark.parametrize("s", [25, 40, 60])
def test_small_part_of_a_row(s):
    # two groups of columns, each tiny on the other's rows; rows in pairs that
    # agree in their large part: their difference in the other columns is tiny
    rng = np.random.default_rng(s)
    n, K = 200, 10
    X = np.zeros((4 * n, 2 * K))
    for g in range(2):
        rows, on, off = slice(2 * n * g, 2 * n * (g + 1)), slice(K * g, K * (g + 1)), slice(K * (1 - g), 2 * K - K * g)
        X[rows, on] = np.repeat(rng.standard_normal((n, K)), 2, axis=0)
        X[rows, off] = 2.0 ** -s * rng.standard_normal((2 * n, K))
    V = np.concatenate([X, -X])
    Q, _, rank = run(V)
    want = reference(V)
    assert rank == 2 * K
    for g in range(2):
        rows, off = slice(2 * n * g, 2 * n * (g + 1)), slice(K * (1 - g), 2 * K - K * g)
        q, r = Q[rows, off].astype(np.longdouble), want[rows, off]
        got, ref = q[::2] - q[1::2], r[::2] - r[1::2]
        tol = 8 * (2 * K + 8) * EPS * np.linalg.cond(V) * np.sqrt((ref ** 2).sum(1))
        err = np.abs(got - ref).max(1)
        assert (err <= tol).all(), (g, float((err / tol).max()))


def test_scores_of_hyperedges_in_small_rows():
    import paper_2511_06600_gb300 as hef
    rng = np.random.default_rng(3)
    n, K = 600, 12
    scale = np.repeat(2.0 ** -np.arange(0, 60, 3.0), n // 20)  # 20 groups of rows
    X = rng.standard_normal((n, K)) * scale[:, None]
    Q, want = check_rows(X)
    edges = [list(rng.choice(n // 20, 3, replace=False) + n // 20 * g) for g in range(20)
             for _ in range(15)]
    H = from_lists(2 * n, edges)
    t = to_dev(H)
    inc = hef.build_incidence(H.n, t["eptr"], t["pins"], t["w"])
    d = torch.zeros(2 * n, hef.padded_ld(K, torch.float64), dtype=torch.float64, device=DEV)
    d[:, :K] = torch.from_numpy(Q).to(DEV)
    R = hef.edge_resistance(inc, d, K)["R"].cpu().numpy()
    inc.check()
    sp2 = np.array([(want[e].max(0) - want[e].min(0)) ** 2 for e in edges])
    ref = (sp2 / sp2.sum(0)).max(1)
    assert (np.abs(R - ref) <= 1e-9 * ref).all(), float((np.abs(R - ref) / ref).max())
