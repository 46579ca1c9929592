"""One coarsening level (hef_coarsen_level) against the CPU oracle, bit for
bit, where its kernels change their way of working: hyperedges at the edges of
the register, one-round, hashed and unhashed forms of the distinct-cluster
search, basis widths at the edges of the columns a lane holds, and column
scales outside the range of the FP32 bounds."""
import numpy as np
import pytest
import torch

from tests._gpu import DEV, to_dev
from tests._hypergraphs import from_lists
from tests.test_gpu_downstream import assert_level_equal, gpu_level, oracle_level

pytestmark = pytest.mark.gpu


def netlist(n, sizes, seed):
    rng = np.random.default_rng(seed)
    edges = [list(rng.choice(n, size=s, replace=False)) for s in sizes]
    edges += [list(rng.choice(n, size=int(rng.integers(2, 5)), replace=False)) for _ in range(n)]
    return from_lists(n, edges, rng.uniform(0.5, 2, size=len(edges)))


def check(H, K, dtype, QH, seed):
    import paper_2511_06600_gb300 as hef
    rng = np.random.default_rng(seed)
    t = to_dev(H)
    inc = hef.build_incidence(H.n, t["eptr"], t["pins"], t["w"])
    R = rng.uniform(0, 1, size=H.m)
    eta = rng.uniform(0, 1, size=H.n) * 1e-3
    Qd = torch.zeros(H.n, hef.padded_ld(K, dtype), dtype=dtype)
    Qd[:, :K] = torch.from_numpy(rng.standard_normal((H.n, K)))
    Qh = Qd[:, :K].numpy()
    got = gpu_level(t, inc, torch.from_numpy(R).to(DEV), torch.from_numpy(eta).to(DEV),
                    Qd.to(DEV), K, torch.from_numpy(QH).to(DEV))
    want = oracle_level(H, R, Qh, QH, eta)
    assert_level_equal(got, want)
    assert (want["target"] >= 0).any()


@pytest.mark.parametrize("sizes", [(7, 8, 9, 31, 32, 33), (64, 65, 511, 512, 513), (800, 544, 2)])
def test_long_hyperedges(sizes):
    check(netlist(900, sizes, sum(sizes)), 12, torch.float32, np.full(12, 0.75), 3)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("K", [1, 31, 64, 65, 128, 129, 256, 257, 512])
def test_basis_widths(K, dtype):
    QH = np.random.default_rng(K).uniform(0.5, 2, size=K)
    QH[K // 2] = 0.0 if K > 1 else 1.0
    check(netlist(150, (40, 9), K), K, dtype, QH, K + 1)


@pytest.mark.parametrize("scale", [1e-290, 1e-31, 1e-29, 1e29, 1e31, 1e200])
def test_column_scales(scale):
    QH = np.random.default_rng(5).uniform(0.5, 2, size=20)
    QH[[2, 7]] *= scale
    check(netlist(150, (40, 9), 6), 20, torch.float64, QH, 7)
