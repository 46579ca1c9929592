"""The staged scoring pass (hef_edge_resistance on rows that a tensor map can
address) at the edges of its column parts, chunks and pin groups, against the
oracle's spreads and ratios on the same Q.

Tolerances: FP64 sums Q_H of m positive terms in another order, (m + 8) eps;
FP32 spreads are exact differences of the same FP32 values up to one rounding,
and Q_H sums at most ~40 FP32 terms before FP64 takes over, so R and Q_H agree
to 64 FP32 eps."""
import numpy as np
import pytest
import torch

from oracle import hef_oracle as O
from tests._gpu import DEV, to_dev
from tests._hypergraphs import from_lists

pytestmark = pytest.mark.gpu


def netlist(n, seed):
    rng = np.random.default_rng(seed)
    sizes = list(rng.integers(2, 6, size=300)) + [12, 13, 31, 32, 33, 63, 64, 65, 100, 1, 0]
    rng.shuffle(sizes)
    edges = [list(rng.choice(n, size=int(s), replace=False)) for s in sizes]
    return from_lists(n, edges, rng.uniform(0.5, 2.0, size=len(edges)))


def check(H, K, dtype, ld, poison=None):
    import paper_2511_06600_gb300 as hef
    rng = np.random.default_rng(K)
    t = to_dev(H)
    inc = hef.build_incidence(H.n, t["eptr"], t["pins"], t["w"])
    Q = torch.full((H.n, ld), float("nan"), dtype=dtype)
    Q[:, :K] = torch.from_numpy(rng.standard_normal((H.n, K)))
    out = hef.edge_resistance(inc, Q.to(DEV), K)
    inc.check()
    Qh = Q[:, :K].numpy()
    sp, pmax, pmin = O.spreads(Qh, H.eptr, H.pins)
    sp64 = sp.astype(np.float64)
    QH = (H.w[:, None] * sp64 ** 2).sum(0)
    ratio = sp64 ** 2 / QH
    tol = (H.m + 8) * np.finfo(np.float64).eps if dtype == torch.float64 else 64 * np.finfo(np.float32).eps
    assert np.abs(out["QH"].cpu().numpy() / QH - 1).max() <= tol
    R = out["R"].cpu().numpy()
    big = np.diff(H.eptr) >= 2
    assert np.abs(R[big] / ratio.max(1)[big] - 1).max() <= tol
    assert (R[~big] == 0).all()
    arg = out["argvec"].cpu().numpy()
    rows = np.arange(H.m)
    assert (ratio[rows[big], arg[big]] >= ratio.max(1)[big] * (1 - tol)).all()
    assert (arg[~big] == -1).all()
    assert np.array_equal(out["pmax"].cpu().numpy()[big], pmax[rows[big], arg[big]])
    assert np.array_equal(out["pmin"].cpu().numpy()[big], pmin[rows[big], arg[big]])


@pytest.mark.parametrize("dtype,K,pad", [
    (torch.float32, 1, 0), (torch.float32, 4, 0), (torch.float32, 31, 0), (torch.float32, 100, 0),
    (torch.float32, 161, 0), (torch.float32, 192, 0), (torch.float32, 193, 0),
    (torch.float32, 300, 4), (torch.float32, 384, 0), (torch.float32, 512, 0),
    (torch.float64, 1, 0), (torch.float64, 20, 0), (torch.float64, 95, 0), (torch.float64, 97, 0),
    (torch.float64, 160, 2), (torch.float64, 257, 0), (torch.float64, 512, 0)])
def test_widths(dtype, K, pad):
    import paper_2511_06600_gb300 as hef
    check(netlist(400, K), K, dtype, hef.padded_ld(K, dtype) + pad)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_few_windows(dtype):
    # fewer windows of pins than CTAs, and a single one
    check(from_lists(5, [[0, 1, 2], [3, 4]]), 24, dtype, 24)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_infinities_and_nan_in_q(dtype):
    # an infinite entry makes its hyperedges' spreads infinite in that column
    # (Q_H too, so the column scores 0 or NaN ratios); a NaN entry takes part in
    # no extremum
    import paper_2511_06600_gb300 as hef
    H = from_lists(6, [[0, 1, 2], [2, 3], [3, 4, 5], [0, 5]])
    t = to_dev(H)
    inc = hef.build_incidence(H.n, t["eptr"], t["pins"], t["w"])
    Q = torch.arange(6 * 8, dtype=dtype).reshape(6, 8).remainder(7) + 1
    Q[1, 3] = float("nan")
    out = hef.edge_resistance(inc, Q.to(DEV), 8)
    Qn = Q.numpy().astype(np.float64)
    QH = np.zeros(8)
    for e in ([0, 1, 2], [2, 3], [3, 4, 5], [0, 5]):
        QH += (np.fmax.reduce(Qn[e]) - np.fmin.reduce(Qn[e])) ** 2
    assert np.allclose(out["QH"].cpu().numpy(), QH, rtol=1e-6)
    Q[4, 2] = float("inf")
    out = hef.edge_resistance(inc, Q.to(DEV), 8)
    assert np.isinf(out["QH"].cpu().numpy()[2])
