"""A batched call leaves the calling thread's launch-form settings as it found
them, in either Krylov form of the batch."""
import pytest
import torch

from netlists.synth import grid_netlist
from tests.test_gpu_batch import batch_inputs

pytestmark = pytest.mark.gpu


def kernels_of_a_call(t, k):
    import paper_2511_06600_gb300 as hef
    torch.cuda.synchronize()
    hef.trace_read()
    hef.trace_kernels("k_")
    try:
        hef.hyperedge_resistance(t["n"], t["eptr"], t["pins"], t["w"], t["x0c"], t["x0b"], k,
                                 torch.float64)
        torch.cuda.synchronize()
    finally:
        hef.trace_kernels(None)
    return set(hef.trace_read())


@pytest.mark.parametrize("batch_form", [0, 1])
@pytest.mark.parametrize("persistent", [0, 1])
def test_batched_call_keeps_the_krylov_form_and_the_elimination(batch_form, persistent):
    import paper_2511_06600_gb300 as hef
    k, S = 8, 4  # K = 64: FP64 eliminates over the grid
    graphs, _ = batch_inputs([grid_netlist(40, 30, 1260, 1), grid_netlist(31, 30, 970, 2)], S)
    b = hef.Batch(graphs, k, S, torch.float64, nstreams=2)
    hef.set_batch_krylov_form(batch_form)
    hef.set_krylov_persistent(persistent)
    try:
        before = kernels_of_a_call(graphs[0], k)
        b.run()
        torch.cuda.synchronize()
        after = kernels_of_a_call(graphs[0], k)
    finally:
        hef.set_batch_krylov_form(1)
        hef.set_krylov_persistent(1)
    assert ("k_krylov_steps" in before) == bool(persistent)
    assert "k_chol_grid" in before
    assert after == before
