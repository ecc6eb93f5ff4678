"""A batch does all its work on the stream it is given (and streams of its own): it
runs, and leaves the capture valid, while a blocking stream of the same context is
being captured, when any use of the legacy default stream is an error."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("use_graph", [1, 0])
def test_batch_beside_a_capture(use_graph):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2004_11227_gb300 import _build
    _build.build()
    from paper_2004_11227_gb300 import cmf, synth
    rt = ctypes.CDLL("libcudart.so.13")
    p = cmf.default_params(2, 2, tol_gap=0.0, max_iter=20, check_every=10, use_graph=use_graph)
    items = [cmf.alloc_binary(synth.random_binary(33, 50, seed=1), p),
             cmf.alloc_potts(synth.random_potts(40, 37, 5, seed=2), p)]
    batch = cmf.Batch(items, p)
    side = torch.cuda.Stream()
    batch.solve(side)  # first launches and attributes
    torch.cuda.synchronize()
    captured, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert rt.cudaStreamCreate(ctypes.byref(captured)) == 0
    assert rt.cudaStreamBeginCapture(captured, 2) == 0  # cudaStreamCaptureModeRelaxed
    try:
        status, res = batch.solve(side)
    finally:
        ended = rt.cudaStreamEndCapture(captured, ctypes.byref(graph))
    assert status == cmf.NOT_CONVERGED and [r["iters"] for r in res] == [20, 20]
    assert ended == 0
    if graph:
        rt.cudaGraphDestroy(graph)
    rt.cudaStreamDestroy(captured)
