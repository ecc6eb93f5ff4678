"""Iterations that run one a launch (a relaxation schedule's, remainders) beside the
launches of several: the states of the kernels that make one a launch throughout, bit
for bit, and not slower than they are."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SCHED = np.linspace(0.5, 1.8, 5)


@pytest.fixture(scope="module")
def cmf():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2004_11227_gb300 import _build
    _build.build()
    from paper_2004_11227_gb300 import cmf as m
    return m


def _binary(cmf, inst, calls, **kw):
    b = cmf.alloc_binary(inst, cmf.default_params(2, 2, **kw))
    cmf.cmf_init_binary(b)
    for n in calls:
        cmf.cmf_iterate_binary(b, n)
    cmf.cmf_eval_binary(b)  # raises if a device wait ran out
    return b.state()


# both sides of the size up to which lone iterations leave the chains (2^20 pixels)
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", [(40, 118), (33, 121), (1030, 1030), (1030, 1031)])
def test_binary_scheduled_iterations(cmf, shape, storage, monkeypatch):
    from paper_2004_11227_gb300 import synth
    inst = synth.random_binary(*shape, seed=7, field_alpha=True)
    for calls in ((3,), (6, 1), (7,), (8,), (12,)):  # all scheduled; 1, 2, 3, 7 beyond
        kw = dict(storage=storage, rho_schedule=SCHED)
        got = _binary(cmf, inst, calls, **kw)
        with monkeypatch.context() as m:
            if shape[1] % 2 == 0:  # rows that are not 16-byte aligned: warp strips
                m.setattr(cmf, "pitch_for", lambda w: (w + 3) // 4 * 4 + 2)
            ref = _binary(cmf, inst, calls, variant=16 if shape[1] % 2 else 4, **kw)
        for k in ref:
            np.testing.assert_array_equal(got[k], ref[k], err_msg=f"{k} {calls}")


# both sides of the size from which two labels' lone iterations leave the rows
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", [(60, 62), (1030, 1030), (41, 61), (1000, 1001), (1030, 1031)])
def test_potts_scheduled_iterations(cmf, shape, storage):
    """Odd widths: against the TMA tiles of the automatic height, which the automatic
    choice runs where the costs are float16 planes (here the same values)."""
    from paper_2004_11227_gb300 import synth
    inst = synth.random_potts(*shape, 2, seed=7, field_alpha=True)
    inst.costs = inst.costs.astype(np.float16).astype(inst.costs.dtype)
    for calls in ((3,), (1, 2), (6, 1), (8,), (12,)):
        out = []
        for kw in (dict(), dict(costs=2) if shape[1] % 2 else dict(variant=2)):
            s = cmf.alloc_potts(inst, cmf.default_params(2, 2, storage=storage,
                                                         rho_schedule=SCHED, **kw))
            cmf.cmf_init_potts(s)
            for n in calls:
                cmf.cmf_iterate_potts(s, n)
            cmf.cmf_eval_potts(s)  # raises if a device wait ran out
            out.append(s.state())
        for k in out[0]:
            np.testing.assert_array_equal(out[0][k], out[1][k], err_msg=f"{k} {calls}")


def _us(f):
    best = 1e9
    for i in range(8):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        f()
        b.record()
        b.synchronize()
        if i > 1:
            best = min(best, a.elapsed_time(b) * 1e3)
    return best


# the rows took 1.14 and 1.09 times as long
@pytest.mark.parametrize("shape,other", [((2048, 2048), 2), ((1024, 1023), 16)])
def test_potts_scheduled_iterations_are_not_slower(cmf, shape, other):
    from paper_2004_11227_gb300 import synth
    inst = synth.random_potts(*shape, 2, seed=7, field_alpha=True)
    n, t = 60, []
    for variant in (0, other):
        p = cmf.default_params(2, 2, storage=1, variant=variant, rho_schedule=np.full(n, 1.9))
        s = cmf.alloc_potts(inst, p)
        cmf.cmf_init_potts(s)
        t.append(_us(lambda: cmf.cmf_iterate_potts(s, n)))
    assert t[0] <= 1.06 * t[1], t


# a chain of one warp took 1.3 times as long in all of these
@pytest.mark.parametrize("shape,storage", [((512, 512), 0), ((1024, 1024), 1), ((512, 513), 0)])
def test_binary_scheduled_iterations_are_not_slower(cmf, shape, storage):
    from paper_2004_11227_gb300 import synth
    inst = synth.random_binary(*shape, seed=7, field_alpha=True)
    n, t = 200, []
    for variant in (0, 16 if shape[1] % 2 else 2):
        p = cmf.default_params(2, 2, storage=storage, variant=variant,
                               rho_schedule=np.full(n, 1.9))
        b = cmf.alloc_binary(inst, p)
        cmf.cmf_init_binary(b)
        t.append(_us(lambda: cmf.cmf_iterate_binary(b, n)))
    assert t[0] <= 1.15 * t[1], t
