"""Which certificate kernel a two-label problem runs: from 2^20 to 2^21 pixels, float32
flows, even widths and ADMM that of the warp strips, which reads no tensor maps (counted
through the fault-injection library, in a process of its own), elsewhere the labels side
by side; the certificates agree with those of rows that are not 16-byte aligned, which
only the strips take, within the roundings of float32 terms."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# height, width, algorithm, storage -> strips
CASES = [(1024, 1024, 2, 0, True), (1025, 2046, 2, 0, True), (1024, 1022, 2, 0, False),
         (1025, 2048, 2, 0, False), (1030, 1030, 2, 1, False), (1030, 1031, 2, 0, False),
         (1030, 1030, 3, 0, False)]

CHILD = r"""
import ctypes, json, sys
import torch
sys.path.insert(0, ROOT)
from paper_2004_11227_gb300 import _build
_build.LIB = _build.LIB_INJECT  # this process loads the injection library only
from paper_2004_11227_gb300 import cmf, synth

count = cmf.lib().cmf_debug_map_encodings
count.restype = ctypes.c_longlong
aligned, out = cmf.pitch_for, []
for H, W, algo, storage, _ in CASES:
    inst, r = synth.random_potts(H, W, 2, seed=3, field_alpha=True), []
    for pitch in (aligned, lambda w: (w + 3) // 4 * 4 + 2):
        cmf.pitch_for = pitch
        s = cmf.alloc_potts(inst, cmf.default_params(algo, 2, storage=storage))
        cmf.cmf_init_potts(s)
        cmf.cmf_iterate_potts(s, 4)
        try:  # first launches, beside the library's short limit
            cmf.cmf_eval_potts(s)
        except cmf.CmfError:
            pass
        n = count()
        r.append([cmf.cmf_eval_potts(s)[:2], count() - n])
    out.append(r)
torch.cuda.synchronize()
print("RESULT " + json.dumps(out))
"""


def test_two_label_certificates():
    import __graft_entry__

    __graft_entry__.build()
    code = f"ROOT = {ROOT!r}\nCASES = {CASES!r}\n" + CHILD
    proc = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True,
                          timeout=600)
    assert proc.returncode == 0, proc.stderr[-3000:]
    line = [x for x in proc.stdout.splitlines() if x.startswith("RESULT ")][-1]
    for case, ((a, maps), (b, _)) in zip(CASES, json.loads(line[len("RESULT "):])):
        assert (maps == 0) == case[4], (case, maps)
        # float32 terms of an energy near 0.3 per pixel, summed in double-float
        assert all(abs(x - y) <= 5e-6 * abs(a[0]) for x, y in zip(a, b)), case
