"""What the library does when the runtime refuses a cooperative launch:
orthonormalisation and Krylov steps take their other form and give the results
of a GPU that runs the grid.  The bounds-checked build brings the condition about
(hef_debug_inject), in a child process that selects it through HEF_LIBRARY."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEAD = "import json, sys\nsys.path.insert(0, %r)\nimport torch\nimport paper_2511_06600_gb300 as hef\n" % ROOT


def child(code):
    from paper_2511_06600_gb300 import build
    env = dict(os.environ, HEF_LIBRARY=build.build(debug=True))
    r = subprocess.run([sys.executable, "-c", HEAD + code], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-4000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


REFUSED = r"""
from netlists import start_block
from netlists.synth import grid_netlist
from tests._gpu import to_dev
out = {}
for dtype, K in ((torch.float64, 64), (torch.float64, 161), (torch.float32, 200)):
    got = []
    for what in (0, 1):
        V = torch.randn(1500, K, generator=torch.Generator().manual_seed(K), dtype=torch.float64)
        d = torch.zeros(1500, hef.padded_ld(K, dtype), dtype=dtype, device="cuda")
        d[:, :K] = V.to(dtype)
        hef.lib().hef_debug_inject(what)
        Q, R, rank = hef.orthonormalize(d, K, want_R=True)
        hef.lib().hef_debug_inject(0)
        got.append((Q.clone(), R, int(rank)))
    out["%s %d" % (dtype, K)] = [got[1][2], bool(torch.equal(got[0][0], got[1][0])),
                                 bool(torch.equal(got[0][1], got[1][1]))]
H = grid_netlist(40, 30, 1260, 1)
t = to_dev(H, *start_block(H.n, H.m, 4, 0))
R = []
for what in (0, 1):
    hef.lib().hef_debug_inject(what)
    R.append(hef.hyperedge_resistance(H.n, t["eptr"], t["pins"], t["w"], t["x0c"], t["x0b"], 8,
                                      torch.float64)["R"])
out["whole"] = float((R[0] - R[1]).abs().max() / R[0].abs().max())
print(json.dumps(out))
"""


def test_refused_grid_takes_the_one_cta_elimination():
    out = child(REFUSED)
    assert out.pop("whole") <= 1e-12  # per-step Krylov sums in another order
    assert len(out) == 3
    for key, (rank, same_q, same_r) in out.items():
        assert rank == int(key.split()[1]) and same_q and same_r, key
