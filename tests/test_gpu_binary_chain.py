"""Binary ADMM by chains of warps (the automatic choice): the states of the
kernels that ran those grids before (even widths: two iterations per launch by
warp strips; odd widths: TMA tiles) bit for bit, and certificates that agree
with the separate certificate kernel.  The certificates sum float32 terms of
equal states in double-float, so they differ by term roundings only: 1e-7 of
the energy (about one last bit of each term) bounds them."""
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


def _run(cmf, inst, algo, calls, **kw):
    b = cmf.alloc_binary(inst, cmf.default_params(algo, 2, **kw))
    assert b.pitch % 4 == (2 if kw.get("variant") == 4 else 0)
    cmf.cmf_init_binary(b)
    for n in calls:
        cmf.cmf_iterate_binary(b, n)
    cmf.cmf_eval_binary(b)  # raises if a device wait ran out
    return b.state()


# strip edges (116 to 124 owned columns, four per lane), odd and ragged widths,
# one row, bands of one row
SHAPES = [(1, 1), (1, 2), (3, 130), (5, 116), (40, 118), (64, 112), (257, 114), (100, 250),
          (2, 57), (33, 121), (130, 61), (7, 233)]


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", SHAPES)
def test_chain_matches_strips_and_tiles(cmf, shape, storage, monkeypatch):
    from paper_2004_11227_gb300 import synth
    H, W = shape
    inst = synth.random_binary(H, W, seed=H + W, field_alpha=H % 2 == 1)
    ref = 16 if W % 2 else 4
    for algo, aniso, calls in ((2, 0, (13,)), (2, 1, (5,)), (1, 0, (1, 2)), (0, 0, (3,)),
                               (4, 0, (4, 1)), (5, 0, (8,))):
        kw = dict(storage=storage, aniso=aniso)
        with monkeypatch.context() as m:
            if ref == 4:  # rows that are not 16-byte aligned: warp strips
                m.setattr(cmf, "pitch_for", lambda w: (w + 3) // 4 * 4 + 2)
            a = _run(cmf, inst, algo, calls, variant=ref, **kw)
        b = _run(cmf, inst, algo, calls, **kw)
        for k in a:
            np.testing.assert_array_equal(a[k], b[k], err_msg=f"{k} algo {algo} aniso {aniso}")


@pytest.mark.parametrize("check_every", [1, 4, 10])
@pytest.mark.parametrize("shape", [(1, 3), (40, 118), (33, 121), (300, 250)])
def test_chain_certificates(cmf, shape, check_every):
    from paper_2004_11227_gb300 import synth
    inst = synth.random_binary(*shape, seed=3, field_alpha=True)
    p = cmf.default_params(2, 2, tol_gap=0.0, max_iter=2 * check_every, check_every=check_every)
    b = cmf.alloc_binary(inst, p)
    status, iters, hist = cmf.cmf_solve_binary(b)
    assert status == cmf.NOT_CONVERGED and iters == 2 * check_every
    E, D, gap, res = cmf.cmf_eval_binary(b)
    assert abs(hist[-1, 1] - E) <= 1e-7 * abs(E)
    assert abs(hist[-1, 2] - D) <= 1e-7 * abs(E)
    assert abs(hist[-1, 4] - res) <= 1e-6 * max(res, 1e-3)


def test_chain_strided_planes(cmf):
    """Padding columns of NaN: neither read nor written."""
    from paper_2004_11227_gb300 import synth
    inst = synth.random_binary(37, 125, seed=5, field_alpha=True)
    out = []
    for pad in (0.0, float("nan")):
        b = cmf.alloc_binary(inst, cmf.default_params(2, 2))
        cmf.cmf_init_binary(b)
        for t in (b.u, b.qx, b.qy, b.ps, b.pt, b.Cs, b.Ct, b.alpha):
            t[..., b.W:] = pad
        cmf.cmf_iterate_binary(b, 9)
        out.append(b.state())
        assert all(bool(torch.isnan(t[..., b.W:]).all()) if pad != pad else
                   bool((t[..., b.W:] == 0).all()) for t in (b.u, b.qx, b.qy, b.ps, b.pt))
    for k in out[0]:
        np.testing.assert_array_equal(out[0][k], out[1][k])
