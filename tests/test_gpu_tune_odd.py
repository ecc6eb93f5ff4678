"""Autotuning at odd widths includes the kernel that the automatic choice runs there."""
import pytest

torch = pytest.importorskip("torch")


@pytest.mark.gpu
def test_tuned_odd_width_runs_the_automatic_kernel():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2004_11227_gb300 import _build
    _build.build()
    from paper_2004_11227_gb300 import cmf, synth
    # twice as fast as any tile kernel at this size
    b = cmf.alloc_binary(synth.config2(901, 1407), cmf.default_params(2, 2, tol_gap=1e-3,
                                                                      max_iter=2000))
    best, ms = cmf.cmf_autotune_binary(b)
    assert best.variant == 0 and ms > 0
