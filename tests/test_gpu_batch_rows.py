"""Batches on the single solves' kernels: Potts instances with the labels side
by side (all label-count classes, even and odd widths), binary ones by chains
of warps.  A batch keeps the roundings its kernels always had (its chunks
complete u in a launch of their own, its binary and odd-width instances follow
the tile and strip kernels), so states are a few last bits from the single
solver's: 30 iterations, values up to 2, about ten roundings each, a
non-expansive iteration: 30 x 10 x 6e-8 x 2 < 4e-5."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(2, 64, 64), (2, 57, 121), (2, 130, 240), (2, 1, 3), (3, 40, 58), (3, 33, 61),
          (4, 64, 112), (8, 48, 90), (8, 90, 57), (6, 30, 130), (16, 40, 64), (11, 20, 77),
          (20, 24, 40), (5, 3, 1)]


@pytest.fixture(scope="module")
def cmf():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2004_11227_gb300 import _build
    _build.build()
    from paper_2004_11227_gb300 import cmf as m
    return m


def _items(cmf, p):
    from paper_2004_11227_gb300 import synth
    out = []
    for k, (L, H, W) in enumerate(SHAPES):
        if L == 2:
            out.append(cmf.alloc_binary(synth.random_binary(H, W, seed=k, field_alpha=k % 2 == 0),
                                        p))
        else:
            out.append(cmf.alloc_potts(synth.random_potts(H, W, L, seed=k,
                                                          field_alpha=k % 2 == 0), p))
    return out


# check intervals with an even and an odd number of pairs, and fewer iterations
# than a chain is long
@pytest.mark.parametrize("check_every", [2, 10, 20])
@pytest.mark.parametrize("rows", [0, 8])
def test_batch_matches_single(cmf, check_every, rows):
    n = 30 // check_every * check_every
    kw = dict(tol_gap=0.0, check_every=check_every, max_iter=n)
    p = cmf.default_params(2, 2, batch_rows=rows, **kw)
    items = _items(cmf, p)
    status, res = cmf.cmf_solve_batch(items, p)
    assert status == cmf.NOT_CONVERGED and all(r["iters"] == n for r in res)
    for (L, H, W), got, k in zip(SHAPES, items, range(len(SHAPES))):
        q = cmf.default_params(2, 2, a2=max(4.0, 2.0 * L), **kw)
        one = _items(cmf, q)[k]
        if L == 2:
            cmf.cmf_init_binary(one)
            cmf.cmf_iterate_binary(one, n)
        else:
            cmf.cmf_init_potts(one)
            for _ in range(n // check_every):
                cmf.cmf_iterate_potts(one, check_every)
        a, b = got.state(), one.state()
        for f in a:
            assert np.abs(a[f] - b[f]).max() <= 4e-5, ((L, H, W), f)


def test_batch_repeated_on_one_workspace(cmf):
    """The tensor maps a batch leaves in its workspace do not reach the next
    batch on the same workspace, whose instances lie elsewhere."""
    p = cmf.default_params(2, 2, tol_gap=0.0, check_every=10, max_iter=20)
    first, second, fresh = _items(cmf, p), _items(cmf, p), _items(cmf, p)
    b1, b2 = cmf.Batch(first, p), cmf.Batch(second, p)
    b1.solve()
    b2.ws = b1.ws
    b2.solve()
    cmf.cmf_solve_batch(fresh, p)
    for x, y in zip(second, fresh):
        a, b = x.state(), y.state()
        for f in a:
            np.testing.assert_array_equal(a[f], b[f])
