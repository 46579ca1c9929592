"""Conditions that the bounds-checked build brings about (hef_debug_inject), in a
child process that selects it through HEF_LIBRARY.

A refused cooperative launch: orthonormalisation and Krylov steps take their
other form and give the results of a GPU that runs the grid.

An expired wait in the last kernel of hef_orthonormalize: every call that runs
it says so."""
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


EXPIRED = r"""
from netlists import start_block
from netlists.synth import grid_netlist
from tests._gpu import to_dev
out = {}
H = grid_netlist(30, 20, 630, 1)
k, S = 5, 2
x0c, x0b = start_block(H.n, H.m, S, 0)
t = to_dev(H, x0c, x0b)
t["n"] = H.n
args = (H.n, t["eptr"], t["pins"], t["w"], t["x0c"], t["x0b"], k)


def status(fn):
    try:
        fn()
        return 0
    except hef.HefError as e:
        return e.status


for name, dtype in (("f64", torch.float64), ("f32", torch.float32)):
    d = torch.randn(500, 20, generator=torch.Generator().manual_seed(1)).to("cuda", dtype)
    pipe = hef.Pipeline(H.n, H.m, H.P, k, S, dtype)
    batch = hef.Batch([t], k, S, dtype, nstreams=1)
    hef.lib().hef_debug_inject(2)
    out[name + " rank"] = int(hef.orthonormalize(d, 20)[2])
    out[name + " whole"] = status(lambda: hef.hyperedge_resistance(*args, dtype))
    pipe.run(*args[1:6])
    out[name + " pipeline"] = status(pipe.check)
    for form in (0, 1):
        hef.set_batch_krylov_form(form)
        batch.run()
        out["%s batch %d" % (name, form)] = status(batch.check)
    starts = lambda lv, n, m: tuple(torch.from_numpy(x).cuda() for x in start_block(n, m, S, lv))
    out[name + " levels"] = status(lambda: hef.multilevel(H.n, t["eptr"], t["pins"], t["w"], starts,
                                                          k, 1, dtype))
    out[name + " host"] = status(lambda: hef.resistance_host(
        H.n, t["eptr"].cpu(), t["pins"].cpu(), t["w"].cpu(), t["x0c"].cpu(), t["x0b"].cpu(), k, dtype))
    for inject in (2, 0):
        hef.lib().hef_debug_inject(inject)
        p = [t[q].clone().requires_grad_() for q in ("w", "x0c", "x0b")]
        R = hef.resistance(*p, H.n, t["eptr"], t["pins"], k, dtype)
        grads = torch.autograd.grad(R, p, torch.ones_like(R))
        # (isolated vertices have the gradient 0 in any case)
        bad = [float(torch.isnan(x).double().mean()) for x in (R, *grads)]
        out["%s gradient %d" % (name, inject)] = -5 if (
            bad[:2] == [1.0, 1.0] and min(bad) > 0.5 if inject else max(bad) == 0) else bad
    out[name + " afterwards"] = -5 if status(lambda: hef.hyperedge_resistance(*args, dtype)) == 0 else 0
    out[name + " rank"] = -5 if out[name + " rank"] == -1 else 0
print(json.dumps(out))
"""


def test_expired_wait_of_the_last_apply_is_reported_by_every_call():
    out = child(EXPIRED)
    assert len(out) == 20
    assert all(v == -5 for v in out.values()), json.dumps(out)
