"""Tensor maps are encoded on the host where a launch first reads them (about 0.15 us
each, beside calls of 30 to 50 us): none in a certificate of the binary model or in a
solve that replays its graph, one buffer set's at most in a call of one iteration.  The
fault-injection library, in a process of its own, counts them."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, json, sys
import torch
sys.path.insert(0, ROOT)
from paper_2004_11227_gb300 import _build
_build.LIB = _build.LIB_INJECT  # this process loads the injection library only
from paper_2004_11227_gb300 import cmf, synth

count = cmf.lib().cmf_debug_map_encodings
count.restype = ctypes.c_longlong
out = {}
for algo in (2, 3):
    for kind in ("binary", "potts"):
        p = cmf.default_params(algo, 2 if kind == "binary" else 4, tol_gap=1e-2, max_iter=200)
        if kind == "binary":
            s = cmf.alloc_binary(synth.random_binary(40, 64, seed=1, field_alpha=True), p)
            it, ev, solve = cmf.cmf_iterate_binary, cmf.cmf_eval_binary, cmf.cmf_solve_binary
        else:
            s = cmf.alloc_potts(synth.random_potts(40, 64, 4, seed=1, field_alpha=True), p)
            it, ev, solve = cmf.cmf_iterate_potts, cmf.cmf_eval_potts, cmf.cmf_solve_potts
        n = []
        try:  # first launches, beside the library's short limit
            solve(s), it(s, 1), it(s, 40), ev(s)
        except cmf.CmfError:
            pass
        for f in (lambda: solve(s), lambda: solve(s), lambda: ev(s), lambda: it(s, 1),
                  lambda: it(s, 40)):
            a = count()
            f()
            n.append(count() - a)
        out[f"{kind}_{algo}"] = n[1:]
torch.cuda.synchronize()
print("RESULT " + json.dumps(out))
"""


def test_maps_are_encoded_where_they_are_read():
    import __graft_entry__

    __graft_entry__.build()
    proc = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + CHILD],
                          capture_output=True, text=True, timeout=600)
    assert proc.returncode == 0, proc.stderr[-3000:]
    line = [x for x in proc.stdout.splitlines() if x.startswith("RESULT ")][-1]
    out = json.loads(line[len("RESULT "):])
    # at most a set's five state planes and the three (binary) or two cost planes, these
    # once a call: replayed solve, certificates, 1 iteration, 40 iterations
    most = {"binary_2": [0, 0, 8, 18], "binary_3": [0, 0, 8, 13],
            "potts_2": [0, 7, 7, 12], "potts_3": [0, 7, 7, 12]}
    for name, counts in out.items():
        assert all(a <= b for a, b in zip(counts, most[name])), (name, counts)
    assert out["binary_2"][3] == 18  # they are counted
