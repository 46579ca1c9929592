"""The one-launch Krylov form on small hypergraphs (few CTAs, ranges that may
be empty, CTAs that own a single row) against the three launches per step:
the same sums in another order.  Tolerances as in the comparison on larger
hypergraphs: 1e-12 (FP64) and 1e-5 (FP32) of the largest score."""
import numpy as np
import pytest
import torch

from netlists import start_block
from netlists.synth import grid_netlist
from tests._gpu import rel_errors, run_pipeline
from tests._hypergraphs import from_lists, random_hypergraph

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def restore_default():
    yield
    import paper_2511_06600_gb300 as hef
    hef.set_krylov_persistent(1)


def both(H, k, S, dtype):
    import paper_2511_06600_gb300 as hef
    x0c, x0b = start_block(H.n, H.m, S, 1)
    out = []
    for form in (1, 0):
        hef.set_krylov_persistent(form)
        out.append(run_pipeline(H, x0c, x0b, k, dtype)["R"])
    return out


@pytest.mark.parametrize("dtype,tol", [(torch.float64, 1e-12), (torch.float32, 1e-5)])
@pytest.mark.parametrize("nx,ny,S", [(8, 8, 1), (12, 11, 2), (40, 32, 4), (64, 63, 8), (97, 91, 4)])
def test_small_netlists(nx, ny, S, dtype, tol):
    H = grid_netlist(nx, ny, int(1.05 * nx * ny), nx + ny)
    a, b = both(H, 3, S, dtype)
    assert rel_errors(a, b)["normwise"] <= tol


def test_one_row_per_range_and_isolated_vertices():
    H = from_lists(200, [[0, 1], [1, 2], [2, 0], [198, 199], [5], []])
    a, b = both(H, 2, 1, torch.float64)
    assert np.abs(a - b).max() <= 1e-12 * b.max()


def test_one_long_hyperedge():
    H = random_hypergraph(300, 40, 5, 3, weights=True)
    H = from_lists(300, [list(range(250))] + [list(H.pins[H.eptr[e]:H.eptr[e + 1]])
                                              for e in range(H.m)])
    a, b = both(H, 4, 2, torch.float64)
    assert rel_errors(a, b)["normwise"] <= 1e-12


def test_calls_on_several_streams_at_once():
    # cooperative launches of different streams and threads take turns
    import threading

    import paper_2511_06600_gb300 as hef
    from tests._gpu import to_dev
    nets = []
    for i in range(4):
        H = grid_netlist(40 + 9 * i, 50, int(1.05 * (40 + 9 * i) * 50), i)
        nets.append((H, to_dev(H, *start_block(H.n, H.m, 2, i))))

    def score(H, t):
        return hef.hyperedge_resistance(H.n, t["eptr"], t["pins"], t["w"], t["x0c"], t["x0b"], 12,
                                        torch.float64)["R"]

    alone = [score(H, t).cpu() for H, t in nets]
    torch.cuda.synchronize()
    got, errors = [None] * 4, []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(5):
                    got[i] = score(*nets[i]).cpu()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors
    for a, b in zip(alone, got):
        assert torch.equal(a, b)
