"""The gradient at basis widths where the QR adjoint's kernels change shape
(columns per CTA round, elements of the lower triangle per CTA): Euler's
identity.  R does not change when every weight is scaled by t and the starts
stay, except through Q_H, which scales with t: sum_e w_e dL/dw_e = -L.  It
holds to rounding of the sums in the adjoints, 1e-9 of |L| in FP64 and 1e-4 in
FP32, for any loss with fixed coefficients."""
import numpy as np
import pytest
import torch

from netlists import start_block
from netlists.synth import grid_netlist
from tests._gpu import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol", [(torch.float64, 1e-9), (torch.float32, 1e-4)])
@pytest.mark.parametrize("nx,ny,k,S", [(20, 18, 1, 1), (31, 17, 4, 2), (40, 39, 8, 1), (60, 50, 4, 8),
                                       (90, 90, 8, 16)])
def test_euler_identity(nx, ny, k, S, dtype, tol):
    import paper_2511_06600_gb300 as hef
    H = grid_netlist(nx, ny, int(1.05 * nx * ny), nx, weight_law="loguniform")
    t = to_dev(H, *start_block(H.n, H.m, S, 2))
    w = t["w"].clone().requires_grad_()
    R = hef.resistance(w, t["x0c"], t["x0b"], H.n, t["eptr"], t["pins"], k, dtype)
    g = torch.from_numpy(np.random.default_rng(1).uniform(0.5, 1.0, H.m)).to(R)
    L = float((g * R.detach()).sum())
    (dw,) = torch.autograd.grad(R, w, g)
    assert abs(float((w.detach() * dw).sum()) + L) <= tol * abs(L)
