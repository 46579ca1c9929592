"""The incidence build at the ends of its division table and with weights at
the ends of the FP32 and FP64 ranges, against numpy (every scalar is one
correctly rounded quotient or a sum of them in incidence order)."""
import numpy as np
import pytest
import torch

from tests._gpu import to_dev
from tests._hypergraphs import from_lists

pytestmark = pytest.mark.gpu


def check(H):
    import paper_2511_06600_gb300 as hef
    t = to_dev(H)
    inc = hef.build_incidence(H.n, t["eptr"], t["pins"], t["w"])
    inc.check()
    out = {k: v.cpu().numpy() for k, v in inc.export().items()}
    size = np.diff(H.eptr)
    first = np.array([H.pins[H.eptr[e]:H.eptr[e + 1]].min() if size[e] else 0 for e in range(H.m)])
    perm = np.lexsort((np.arange(H.m), first))
    assert np.array_equal(out["perm"], perm)
    deg = np.bincount(H.pins, minlength=H.n)
    assert np.array_equal(out["vptr"], np.concatenate(([0], np.cumsum(deg))))
    rank = np.empty(H.m, dtype=np.int64)
    rank[perm] = np.arange(H.m)
    edge_of = np.repeat(np.arange(H.m), size)
    order = np.lexsort((rank[edge_of], H.pins))
    assert np.array_equal(out["vedge"], edge_of[order])
    k = size.astype(np.float64)
    on = size >= 2
    wh = np.where(on, H.w / np.where(on, k - 1, 1), 0.0)
    term = np.where(on, wh * (k - 1), 0.0)
    z = np.where(on, H.w / np.maximum(k, 1), 0.0)
    dc, db = np.zeros(H.n), np.zeros(H.n)
    for v, e in zip(H.pins[order], edge_of[order]):
        dc[v] += term[e]
        db[v] += z[e]
    assert np.array_equal(out["dc"], dc) and np.array_equal(out["db"], db)
    return inc


@pytest.mark.parametrize("seed", [1, 2])
def test_sizes_around_the_tables(seed):
    rng = np.random.default_rng(seed)
    sizes = [0, 1, 2, 3, 4, 5, 7, 8, 9, 31, 32, 33, 62, 63, 64, 65, 66, 100, 128, 129]
    edges = [list(rng.choice(400, size=s, replace=False)) for s in sizes]
    edges += [list(rng.choice(400, size=int(rng.integers(2, 7)), replace=False)) for _ in range(9000)]
    check(from_lists(400, edges, rng.uniform(0.1, 3, size=len(edges))))


@pytest.mark.parametrize("w", [5e-324, 1e-310, 1e-300, 1e-45, 3.3e-39, 1.1e38, 3.5e38, 1e300, 1e307])
def test_weights_at_the_ends_of_the_ranges(w):
    rng = np.random.default_rng(3)
    edges = [list(rng.choice(60, size=int(s), replace=False)) for s in rng.integers(2, 20, size=40)]
    check(from_lists(60, edges, w * rng.uniform(1, 1.3, size=40)))
