"""Binary rPDRQ on shared TMA rows (the automatic choice on even widths, one
sweep): every width and band gives the states of the one-warp strips, which ran
those grids before it, bit for bit."""
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
    s = cmf.alloc_binary(inst, cmf.default_params(cmf.RPDRQ, 2, **kw))
    cmf.cmf_init_binary(s)
    if pad is not None:
        for t in (s.u, s.qx, s.qy, s.ps, s.pt, s.Cs, s.Ct, s.alpha):
            t[..., s.W:] = pad
    for n in calls:
        cmf.cmf_iterate_binary(s, n)
    cmf.cmf_eval_binary(s)  # raises if a device wait ran out
    return s.state()


# strip (56 owned columns) and block (224) edges, one row, bands shorter and
# longer than the rings
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", [(1, 2), (2, 56), (7, 58), (33, 112), (64, 222), (5, 224),
                                   (131, 226), (700, 240), (3000, 62)])
def test_rows_match_strips(cmf, shape, storage):
    from paper_2004_11227_gb300 import synth
    H, W = shape
    inst = synth.random_binary(H, W, seed=H + W, field_alpha=H % 2 == 1)
    for aniso, calls in ((0, (7,)), (1, (1, 2))):
        kw = dict(storage=storage, aniso=aniso)
        got, ref = (_run(cmf, inst, calls, variant=v, **kw) for v in (0, 2))
        for k in ref:
            assert np.isfinite(got[k]).all()
            np.testing.assert_array_equal(got[k], ref[k], err_msg=f"{k} aniso={aniso}")


def test_padding_is_not_read(cmf):
    """NaN in the columns between the width and the pitch."""
    from paper_2004_11227_gb300 import synth
    inst = synth.random_binary(37, 70, seed=5, field_alpha=True)
    a, b = (_run(cmf, inst, (5,), pad=v) for v in (0.0, float("nan")))
    for k in a:
        np.testing.assert_array_equal(a[k], b[k])
