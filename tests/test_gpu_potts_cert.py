"""Potts certificates with the labels side by side against the FP64 oracle, at
strip edges, odd widths, single rows and the ends of the label-count classes.

Tolerance: float32 per-pixel terms (about ten roundings of values up to 2 for
an energy near 0.3 per pixel: 10 x 6e-8 x 2 / 0.3 < 5e-6) summed in
double-float; the residual is a norm of differences of values near 1, each a
few last bits off (1e-6 of sqrt(pixels x labels))."""
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


@pytest.mark.parametrize("algo", [2, 3])
@pytest.mark.parametrize("shape", [(1, 1, 2), (1, 2, 3), (5, 61, 2), (33, 60, 4), (40, 121, 5),
                                   (64, 64, 8), (100, 130, 11), (37, 90, 16), (130, 61, 7)])
def test_potts_certificates(cmf, orc, shape, algo):
    from paper_2004_11227_gb300 import synth
    H, W, L = shape
    inst = synth.random_potts(H, W, L, seed=H + W, field_alpha=H % 2 == 0)
    for storage, aniso, n in ((0, 0, 7), (0, 1, 40), (1, 0, 7), (2, 0, 3)):
        p = cmf.default_params(algo, L, storage=storage, aniso=aniso)
        s = cmf.alloc_potts(inst, p)
        cmf.cmf_init_potts(s)
        cmf.cmf_iterate_potts(s, n)
        E, D, gap, res = cmf.cmf_eval_potts(s)
        e, d, g, r = orc.potts_eval(inst.costs, inst.alpha, s.state(),
                                    orc.default_params(algo, L, aniso=aniso))
        assert abs(E - e) <= 5e-6 * abs(e) and abs(D - d) <= 5e-6 * abs(e)
        assert abs(res - r) <= 1e-6 * np.sqrt(H * W * L)


def test_potts_certificates_padding(cmf):
    """Padding columns of NaN do not enter."""
    from paper_2004_11227_gb300 import synth
    inst = synth.random_potts(37, 71, 3, seed=5, field_alpha=True)
    out = []
    for pad in (0.0, float("nan")):
        s = cmf.alloc_potts(inst, cmf.default_params(2, 3))
        cmf.cmf_init_potts(s)
        for t in (s.u, s.qx, s.qy, s.p, s.ps, s.C, s.alpha):
            t[..., s.W:] = pad
        out.append(cmf.cmf_eval_potts(s))
    assert out[0] == out[1]
