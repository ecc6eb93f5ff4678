"""The smallest workspace a batch accepts does not grow: what held the tile and
strip kernels' tables and states before the kernels with tensor maps existed
(sizes pinned from then) is still enough, by the kernels that need no maps."""
import ctypes

import pytest

# (instances, algorithm, params.batch_rows) -> bytes
SIZES = {(1, 2, 0): 124672,
         (12, 2, 0): 86067200,
         (12, 2, 8): 86077696,
         (12, 3, 0): 86065664,
         (12, 4, 0): 86067200,
         (64, 2, 24): 1011460352,
         (256, 2, 12): 4203145984}


def _instances(cmf, n, alloc):
    insts = (cmf.Instance * n)()
    for k in range(n):
        i = insts[k]
        i.L = (2, 3, 4, 8)[k % 4]
        i.model = int(i.L > 2)
        i.H = 64 + 37 * (k % 20)
        i.W = i.H + k % 3
        i.pitch = (i.W + 1 + 31) // 32 * 32
        i.alpha0 = 0.3
        alloc(i)
    return insts


@pytest.mark.parametrize("key", list(SIZES))
def test_smallest_workspace(key):
    from paper_2004_11227_gb300 import _build
    _build.build()
    from paper_2004_11227_gb300 import cmf
    torch = pytest.importorskip("torch")
    if torch.cuda.is_available():
        pytest.skip("the buffers are not real: sizes only, without a GPU")
    n, algo, rows = key
    buf = ctypes.create_string_buffer(1 << 16)
    ptr = (ctypes.addressof(buf) + 255) // 256 * 256

    def alloc(i):
        i.d_cost = i.d_u = i.d_qx = i.d_qy = i.d_p = i.d_ps = ptr

    insts = _instances(cmf, n, alloc)
    q = cmf.default_params(algo, 2, batch_rows=rows, check_every=10, max_iter=1000)

    def solve(size):
        return cmf.lib().cmf_solve_batch(insts, n, ctypes.byref(q), ptr, ctypes.c_size_t(size),
                                         None)

    assert solve(SIZES[key] - 1) == cmf.ENOMEM
    assert solve(SIZES[key]) == cmf.ECUDA  # accepted; then there is no GPU


@pytest.mark.gpu
def test_smallest_workspace_solves():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2004_11227_gb300 import _build
    _build.build()
    from paper_2004_11227_gb300 import cmf
    n, keep, states = 12, [], []

    def alloc(i):
        g = torch.Generator(device="cuda").manual_seed(i.H)
        C = torch.rand((i.L, i.H, i.pitch), device="cuda", generator=g)
        s = [torch.zeros((k, i.H, i.pitch), device="cuda") for k in (i.L, i.L, i.L, i.L, 1)]
        if i.model == 0:
            s = [torch.zeros((1, i.H, i.pitch), device="cuda") for _ in range(5)]
        keep.append(C)
        states.append(s)
        i.d_cost = C.data_ptr()
        i.d_u, i.d_qx, i.d_qy, i.d_p, i.d_ps = (t.data_ptr() for t in s)

    out = []
    q = cmf.default_params(2, 2, check_every=10, max_iter=20, tol_gap=0.0)
    for full in (True, False):
        states.clear()
        insts = _instances(cmf, n, alloc)
        size = cmf.lib().cmf_batch_workspace_bytes(insts, n, ctypes.byref(q)) if full \
            else SIZES[(12, 2, 0)]
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        status = cmf.lib().cmf_solve_batch(insts, n, ctypes.byref(q), ws.data_ptr(),
                                           ctypes.c_size_t(size), None)
        assert status == cmf.NOT_CONVERGED
        torch.cuda.synchronize()
        out.append([s[0].clone() for s in states])
    # 20 iterations, values up to 2, about ten roundings each, a non-expansive
    # iteration: 20 x 10 x 6e-8 x 2 < 4e-5
    for i, a, b in zip(insts, *out):
        assert float((a[..., :i.W] - b[..., :i.W]).abs().max()) <= 4e-5
