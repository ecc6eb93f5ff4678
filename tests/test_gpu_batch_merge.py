"""Batch blocks that take several base bands, as many as the instances still
active call for: the same iterations and states bit for bit as with one band a
block (batch_rows = 8), while instances retire at different checks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("count", [2, 40])
def test_merged_bands_give_the_same_solution(count, use_graph):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2004_11227_gb300 import _build
    _build.build()
    from paper_2004_11227_gb300 import cmf, synth
    # three classes of label counts, heights that no band height divides
    insts = [synth.potts_shapes(149 + 11 * (k % 9), 60 + 37 * (k % 5), (3, 8, 12)[k % 3],
                                seed=300 + k) for k in range(count)]
    out = []
    for rows in (8, 0):
        p = cmf.default_params(2, 2, tol_gap=1e-3, max_iter=400, check_every=20,
                               batch_rows=rows, use_graph=use_graph)
        items = [cmf.alloc_potts(i, p) for i in insts]
        _, res = cmf.cmf_solve_batch(items, p)
        out.append(([(r["iters"], r["status"]) for r in res], [it.state() for it in items]))
    assert out[0][0] == out[1][0]
    for a, b in zip(out[0][1], out[1][1]):
        for k in a:
            np.testing.assert_array_equal(a[k], b[k])
