"""Grids whose bands are tens of rows high, so that every ring of the row kernels goes
round many times, above all at odd widths (roundings, shares and last columns of their
own): the states of the kernels that ran those grids before, bit for bit, and fused
certificates that agree with the certificate kernel's."""
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


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", [(721, 1283, 8), (1500, 601, 3), (1500, 601, 16),
                                   (1500, 602, 4), (1300, 602, 11)])
def test_potts(cmf, shape, storage):
    """Odd widths: against the TMA tiles of the automatic height, which the automatic
    choice runs where the costs are float16 planes (here the same values)."""
    from paper_2004_11227_gb300 import synth
    H, W, L = shape
    inst = synth.random_potts(H, W, L, seed=H + L, field_alpha=L % 2 == 1)
    inst.costs = inst.costs.astype(np.float16).astype(inst.costs.dtype)
    for algo, aniso, calls in ((2, 0, (7,)), (2, 1, (4,)), (1, 0, (1, 4))):
        out = []
        for kw in (dict(), dict(costs=2) if W % 2 else dict(variant=2)):
            s = cmf.alloc_potts(inst, cmf.default_params(algo, L, storage=storage, aniso=aniso,
                                                         **kw))
            cmf.cmf_init_potts(s)
            for n in calls:
                cmf.cmf_iterate_potts(s, n)
            cmf.cmf_eval_potts(s)  # raises if a device wait ran out
            out.append(s.state())
        for k in out[0]:
            np.testing.assert_array_equal(out[0][k], out[1][k], err_msg=f"{k} {algo} {aniso}")


@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("shape", [(901, 1407), (3000, 301), (2500, 602)])
def test_binary(cmf, shape, storage, monkeypatch):
    from paper_2004_11227_gb300 import synth
    H, W = shape
    inst = synth.random_binary(H, W, seed=H, field_alpha=True)
    for algo, aniso, calls in ((2, 0, (13,)), (2, 1, (5,)), (1, 0, (8, 3)), (4, 0, (8,)),
                               (5, 0, (7,))):
        out = []
        for variant in (0, 16 if W % 2 else 4):
            with monkeypatch.context() as m:
                if variant == 4:  # rows that are not 16-byte aligned: warp strips
                    m.setattr(cmf, "pitch_for", lambda w: (w + 3) // 4 * 4 + 2)
                b = cmf.alloc_binary(inst, cmf.default_params(algo, 2, storage=storage,
                                                              aniso=aniso, variant=variant))
            cmf.cmf_init_binary(b)
            for n in calls:
                cmf.cmf_iterate_binary(b, n)
            cmf.cmf_eval_binary(b)  # raises if a device wait ran out
            out.append(b.state())
        for k in out[0]:
            np.testing.assert_array_equal(out[0][k], out[1][k], err_msg=f"{k} {algo} {aniso}")


# float32 terms of equal states, summed in double-float: about one last bit of each
@pytest.mark.parametrize("shape", [(901, 1407), (3000, 301), (2500, 602)])
def test_binary_certificates(cmf, shape):
    from paper_2004_11227_gb300 import synth
    inst = synth.random_binary(*shape, seed=3, field_alpha=True)
    p = cmf.default_params(2, 2, tol_gap=0.0, max_iter=20, check_every=10)
    b = cmf.alloc_binary(inst, p)
    status, iters, hist = cmf.cmf_solve_binary(b)
    assert status == cmf.NOT_CONVERGED and iters == 20 and len(hist) == 2
    E, D, gap, res = cmf.cmf_eval_binary(b)
    assert abs(hist[-1, 1] - E) <= 1e-7 * abs(E)
    assert abs(hist[-1, 2] - D) <= 1e-7 * abs(E)
    assert abs(hist[-1, 4] - res) <= 1e-6 * max(res, 1e-3)
