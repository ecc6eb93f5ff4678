"""Potts rPDRQ with the labels side by side (the automatic choice on even
widths): every width, band and label count gives the states of the warp strips,
which ran those grids before it, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cmf():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2004_11227_gb300 import _build
    _build.build()
    from paper_2004_11227_gb300 import cmf as m
    return m


def _run(cmf, inst, calls, pad=None, **kw):
    s = cmf.alloc_potts(inst, cmf.default_params(cmf.RPDRQ, inst.L, **kw))
    cmf.cmf_init_potts(s)
    if pad is not None:
        for t in (s.u, s.qx, s.qy, s.p, s.ps, s.C, s.alpha):
            t[..., s.W:] = pad
    for n in calls:
        cmf.cmf_iterate_potts(s, n)
    cmf.cmf_eval_potts(s)  # raises if a device wait ran out
    return s.state()


# strip and band edges (56 owned columns), one row, bands shorter and longer than
# the rings, label counts at the ends of the three block sizes (4, 8, 16)
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", [(1, 2, 2), (2, 56, 3), (7, 58, 4), (3, 112, 5), (64, 64, 8),
                                   (33, 114, 9), (5, 120, 15), (131, 62, 16), (700, 240, 2)])
def test_rows_match_strips(cmf, shape, storage):
    from paper_2004_11227_gb300 import synth
    H, W, L = shape
    inst = synth.random_potts(H, W, L, seed=H + W + L, field_alpha=H % 2 == 1)
    for aniso, calls in ((0, (7,)), (1, (1, 2))):
        kw = dict(storage=storage, aniso=aniso)
        got, ref = (_run(cmf, inst, calls, variant=v, **kw) for v in (0, 2))
        for k in ref:
            assert np.isfinite(got[k]).all()
            np.testing.assert_array_equal(got[k], ref[k], err_msg=f"{k} aniso={aniso}")


def test_padding_is_not_read(cmf):
    """NaN in the columns between the width and the pitch."""
    from paper_2004_11227_gb300 import synth
    inst = synth.random_potts(37, 70, 3, seed=5, field_alpha=True)
    a, b = (_run(cmf, inst, (5,), pad=v) for v in (0.0, float("nan")))
    for k in a:
        np.testing.assert_array_equal(a[k], b[k])
