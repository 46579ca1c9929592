"""The elimination over the whole grid (k_chol_grid, single calls) and in one
CTA (k_chol_aug, inside a batch) do the same operations on every element: a
batch with per-step Krylov launches gives the single calls' bits at basis
widths on both sides of the line between the two."""
import numpy as np
import pytest
import torch

from netlists.synth import grid_netlist
from tests._gpu import run_pipeline
from tests.test_gpu_batch import batch_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,k,S", [(torch.float64, 23, 1), (torch.float64, 6, 4),
                                       (torch.float64, 8, 4), (torch.float64, 25, 1),
                                       (torch.float64, 20, 4), (torch.float32, 20, 4),
                                       (torch.float32, 12, 8), (torch.float32, 21, 4)])
def test_batch_equals_single_calls_bitwise(dtype, k, S):
    import paper_2511_06600_gb300 as hef
    Hs = [grid_netlist(nx, ny, int(1.05 * nx * ny), 7 + nx, weight_law="loguniform")
          for nx, ny in ((80, 75), (61, 50))]
    graphs, host = batch_inputs(Hs, S)
    b = hef.Batch(graphs, k, S, dtype, nstreams=2)
    hef.set_batch_krylov_form(0)
    hef.set_krylov_persistent(0)  # per-step Krylov launches in the single calls too
    try:
        out = b.run()
        torch.cuda.synchronize()
        b.check()
        refs = [run_pipeline(H, x0c, x0b, k, dtype) for H, x0c, x0b in host]
    finally:
        hef.set_batch_krylov_form(1)
        hef.set_krylov_persistent(1)
    for got, ref in zip(out, refs):
        for key in ("R", "QH", "argvec", "pmax", "pmin"):
            assert np.array_equal(got[key].cpu().numpy(), ref[key]), key
