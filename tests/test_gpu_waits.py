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


SERVED = r'''
import ctypes, json, sys
import torch
sys.path.insert(0, sys.argv[1])
from paper_1704_02745_gb300 import inputs, pb

lib = pb.load()
for f in (lib.pb_test_abandon_waits, lib.pb_test_abandon_sums, lib.pb_test_fail_allocs):
    f.argtypes = [ctypes.c_int]
probs = [inputs.random_small(60 + k, *s, n_atoms=12) for k, s in
         enumerate([(33, 20, 29), (40, 17, 33), (25, 26, 27), (61, 33, 45), (2060, 5, 7)])]
out = {}
torch.cuda.set_device(0)
with pb.Context(0) as ctx:
    for prec, tol in (("f32_refine", 1e-9), ("f32", 1e-6)):
        opts = dict(precision=prec, tol=tol, inner_tol=1e-4, warm_start=False)
        def served(srv, which):
            tk = [srv.submit(k, probs[k].grid, probs[k].atoms) for k in which]
            return [(r.status, r.energy, r.info.iterations) for r in (srv.poll(t, 60000)[0] for t in tk)]
        with pb.Server(ctx, 4 << 30, poll_every=8, **opts) as srv:
            ticks = served(srv, range(5))
        with pb.Server(ctx, 4 << 30, **opts) as srv:
            # no memory for the words that CTAs exchange: ticks, for that solve only
            srv.profile_begin()
            served(srv, [0])
            srv.profile_end()
            lib.pb_test_fail_allocs(1)
            no_memory = served(srv, [0])
            lib.pb_test_fail_allocs(0)
            chip = served(srv, range(5))
            lib.pb_test_abandon_sums(1)
            alone = served(srv, [0])
            lib.pb_test_abandon_sums(1)
            together = served(srv, range(5))
            lib.pb_test_abandon_sums(0)
            again = served(srv, range(5))
        out[prec] = dict(ticks=ticks, chip=chip, no_memory=no_memory, alone=alone, together=together, again=again)
    # one grid: the same words
    with pb.Grid(ctx, probs[0].grid, probs[0].atoms) as g:
        phi = torch.zeros(probs[0].grid.shape, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        def solve(poll):
            info = g.solve(phi, check=False, precision="f32_refine", tol=1e-9, inner_tol=1e-4, poll_every=poll)
            return [info.status, g.energy(phi), info.iterations]
        ticks = solve(8)
        lib.pb_test_fail_allocs(1)
        no_memory = solve(0)
        lib.pb_test_fail_allocs(0)
        chip = solve(0)
        out["grid"] = [ticks, no_memory, chip]
print("RESULT " + json.dumps(out))
'''


def test_served_and_short_of_memory():
    out = run(SERVED)
    for prec in ("f32_refine", "f32"):
        o = out[prec]
        bound = 2e-5 if prec == "f32" else 2e-7  # two solves, each within the bound above
        assert all(r[0] == 0 for k in o for r in o[k]), o
        assert o["chip"][4] == o["ticks"][4] and o["chip"][0] != o["ticks"][0], o  # (two forms; the last grid: ticks)
        # given up once, or without memory: the tick form's own result, bit for bit; then the own form again
        assert o["no_memory"] == o["alone"] == [o["ticks"][0]], o
        assert o["again"] == o["chip"], o
        for got, own, tick in zip(o["together"], o["chip"], o["ticks"]):
            assert got in (own, tick) and abs(got[1] - own[1]) <= bound * abs(own[1]), o
        assert o["together"] != o["chip"], o
    ticks, no_memory, chip = out["grid"]
    assert ticks[0] == 0 and no_memory == ticks and chip[0] == 0 and chip != ticks, out["grid"]
