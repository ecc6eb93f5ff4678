"""A bounded wait that runs out in a kernel of the automatic choice, or in a batch, is
reported as CMF_ETIMEOUT, stops the solve at its next check and leaves the context
usable: the fault-injection library (see test_gpu_failure.py) makes every barrier that
waits for input rows expect 16 bytes more than its copies deliver."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OK, ETIMEOUT = 0, 4

CHILD = r"""
import ctypes, json, sys, time
import numpy as np
import torch
sys.path.insert(0, ROOT)
from paper_2004_11227_gb300 import _build
_build.LIB = _build.LIB_INJECT  # this process loads the injection library only
from paper_2004_11227_gb300 import cmf, synth

lib = cmf.lib()
lib.cmf_debug_inject_row_tx.argtypes = [ctypes.c_uint]
lib.cmf_debug_inject_row_tx.restype = ctypes.c_int

def inject(n):
    torch.cuda.synchronize()
    assert lib.cmf_debug_inject_row_tx(n) == 0

class Problem:
    def __init__(self, kind, L, H, W, algo, use_graph):
        p = cmf.default_params(algo, L, tol_gap=1e-3, max_iter=400, check_every=10,
                               use_graph=use_graph)
        self.kind = kind
        self.s = (cmf.alloc_binary(synth.random_binary(H, W, seed=5, field_alpha=True), p)
                  if kind == "binary" else
                  cmf.alloc_potts(synth.random_potts(H, W, L, seed=5, field_alpha=True), p))

    def _call(self, what, *mid):
        s = self.s
        return getattr(lib, f"cmf_{what}_{self.kind}")(
            *s._common(), *mid, cmf._ptr(s.ws), s.ws.numel(), cmf._stream(None))

    def solve(self):
        hist, it = np.zeros((64, 5)), ctypes.c_int(0)
        st = self._call("solve", *self.s._state_ptrs(), hist.ctypes.data_as(ctypes.c_void_p), 64,
                        ctypes.byref(it))
        return st, it.value, hist.tolist()

    def iterate(self, n):
        return self._call("iterate", n, *self.s._state_ptrs())

    def eval(self):
        return self._call("eval", *self.s._state_ptrs(), (ctypes.c_double * 4)())

out = {}
for name, args in CASES.items():
    q = Problem(*args)
    q.solve()  # first launches, beside the library's short limit
    before = q.solve()
    inject(16)
    st, it, _ = q.solve()
    r = {"before": before[0], "solve": st, "iterations": it, "iterate": q.iterate(5)}
    inject(0)
    r["evals"] = [q.eval(), q.eval()]
    if q.kind == "potts":
        inject(16)
        r["eval_itself"] = q.eval()
        inject(0)
    after = q.solve()
    r["after_equal"] = after == before
    out[name] = r

for use_graph in (1, 0):
    p = cmf.default_params(2, 2, tol_gap=1e-3, max_iter=10000000, check_every=10,
                           use_graph=use_graph)
    items = [cmf.alloc_binary(synth.random_binary(40, 60, seed=1), p)]
    items += [cmf.alloc_potts(synth.random_potts(33 + L, 50 + L, L, seed=L), p)
              for L in (3, 4, 7, 12)]
    b = cmf.Batch(items, p)
    def run():
        st = lib.cmf_solve_batch(b.insts, len(items), ctypes.byref(p), cmf._ptr(b.ws),
                                 b.ws.numel(), cmf._stream(None))
        return [st] + [[d.status, d.iters, d.gap] for d in b.insts]
    run()
    before = run()
    inject(16)
    failed = run()
    inject(0)
    out[f"batch_{use_graph}"] = {"before": before[0], "solve": failed[0],
                                 "items": [x[:2] for x in failed[1:]],
                                 "after_equal": run() == before}
torch.cuda.synchronize()
print("RESULT " + json.dumps(out))
"""

# kind, labels, height, width, algorithm, device-driven loop
CASES = {
    "potts_one_service_warp": ("potts", 4, 40, 60, 2, 1),
    "potts_two_service_warps": ("potts", 9, 40, 60, 2, 1),
    "potts_host_loop": ("potts", 6, 40, 60, 2, 0),
    "potts_rpdrq": ("potts", 5, 40, 60, 3, 1),
    "binary_chains": ("binary", 2, 64, 130, 2, 1),
    "binary_chains_odd": ("binary", 2, 41, 61, 2, 1),
    "binary_host_loop": ("binary", 2, 40, 60, 2, 0),
    "binary_rpdrq": ("binary", 2, 40, 60, 3, 1),
}


@pytest.fixture(scope="module")
def result():
    import __graft_entry__

    __graft_entry__.build()
    code = f"ROOT = {ROOT!r}\nCASES = {CASES!r}\n" + CHILD
    # a batch that ran on to its iteration limit would take hours
    proc = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True,
                          timeout=600)
    assert proc.returncode == 0, proc.stderr[-3000:]
    line = [x for x in proc.stdout.splitlines() if x.startswith("RESULT ")][-1]
    return json.loads(line[len("RESULT "):])


@pytest.mark.parametrize("case", list(CASES))
def test_default_kernels_report_a_timeout(result, case):
    r = result[case]
    assert r["before"] == OK
    # stopped at the first check
    assert r["solve"] == ETIMEOUT and (r["iterations"] == 10 or CASES[case][5] == 0)
    # iterate does not synchronise: the next certificate call reports it, once
    assert r["iterate"] == OK and r["evals"] == [ETIMEOUT, OK]
    assert r.get("eval_itself", ETIMEOUT) == ETIMEOUT
    assert r["after_equal"]  # the same history bit for bit


@pytest.mark.parametrize("use_graph", [1, 0])
def test_batch_stops_at_its_next_check(result, use_graph):
    r = result[f"batch_{use_graph}"]
    assert r["before"] == OK and r["solve"] == ETIMEOUT
    assert r["items"] == [[ETIMEOUT, 10]] * 5
    assert r["after_equal"]
