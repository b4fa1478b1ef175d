"""Both bounded waits of the solves, each on its own switch of the fault-test
library (a separate process; nothing faults or hangs):

* pb_test_abandon_sums(n): the next n first grid-wide sums of the resident form
  give up.  Expected: the solve starts over in phase ticks and succeeds.
* pb_test_abandon_waits(n), with poll_every > 0 (phase ticks from the start): the
  next n first-plane stage waits give up.  Expected: PB_ERR_TIMEOUT, and a clean
  next solve.

Energies against the oracle's at 1e-7, the fault tests' bound."""
import json
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r'''
import ctypes, json, sys
import torch
sys.path.insert(0, sys.argv[1])
import oracle
from paper_1704_02745_gb300 import inputs, pb

lib = pb.load()
for f in (lib.pb_test_abandon_waits, lib.pb_test_abandon_sums):
    f.argtypes = [ctypes.c_int]
p = inputs.small_33()
s = oracle.setup(p.grid, p.atoms)
e_ref = oracle.energy(s, oracle.pcg(s, tol=1e-10).phi)
rel = lambda e: abs(e - e_ref) / abs(e_ref)
out = {}
torch.cuda.set_device(0)
with pb.Context(0) as ctx:
    for prec, tol in (("f32_refine", 1e-9), ("f64", 1e-9), ("f32", 1e-6)):
        with pb.Grid(ctx, p.grid, p.atoms) as g:
            phi = torch.zeros(p.grid.shape, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            def solve(poll, warm=False):
                info = g.solve(phi, check=False, precision=prec, tol=tol, poll_every=poll, warm_start=warm)
                return [info.status, rel(g.energy(phi)), info.iterations]
            ticks = solve(8)
            lib.pb_test_abandon_sums(1)
            first = solve(0)
            lib.pb_test_abandon_sums(3)
            out[prec + "_warm"] = [solve(0, True), solve(0, True)]
            lib.pb_test_abandon_sums(0)
            out[prec + "_sum"] = [first, ticks]
            lib.pb_test_abandon_waits(1)
            out[prec + "_wait"] = solve(8)[0]
            lib.pb_test_abandon_waits(0)
            out[prec + "_clean"] = [solve(8), solve(0)]
print("RESULT " + json.dumps(out))
'''


def run(script):
    from paper_1704_02745_gb300 import build
    env = dict(os.environ, PB_LIBRARY=build.build_fault_test())
    r = subprocess.run([sys.executable, "-c", script, ROOT], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    line = [ln for ln in r.stdout.splitlines() if ln.startswith("RESULT ")][-1]
    return json.loads(line[len("RESULT "):])


def test_single_grid():
    out = run(SCRIPT)
    TIMEOUT = 7
    for prec in ("f32_refine", "f64", "f32"):
        bound = 1e-5 if prec == "f32" else 1e-7  # (plain FP32 to 1e-6)
        first, ticks = out[prec + "_sum"]
        assert first[0] == 0 and first[1:] == ticks[1:], out  # the tick form's own result, bit for bit
        for st, err, _ in [first] + out[prec + "_warm"] + out[prec + "_clean"]:
            assert st == 0 and err <= bound, out
        assert out[prec + "_wait"] == TIMEOUT, out
