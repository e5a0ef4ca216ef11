"""kubo_bloch in FP64 with a caller's workspace of kubo_workspace_size() bytes, which knows nothing of the list's length.

Both forms of the sum: bound N_R terms of a column's largest basis entry, each 2^-48 (the FP64-pipe chain's).
The bytes behind the workspace stay as they were.
"""
import ctypes

import numpy as np
import pytest
import tbgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,half,chunk,n", [
    (16, 2, 1024, 40_000),   # slices cut to what is left of 36 MB
    (33, 1, 512, 20_000),
    (4, 2, 256, 100_000),    # two column tiles: a sub-batch that leaves SMs idle gives way to the FP64-pipe kernel
    (16, 2, 1, 3000),        # no room for slices
    (64, 2, 64, 700),
])
def test_workspace_of_the_size_query(W, half, chunk, n):
    import torch
    import paper_2309_06675_gb300 as kubo
    m = tbgen.random_tb(W, half, 1.5, seed=W)
    mesh = (41, 13, 9)
    kidx = torch.from_numpy(np.random.default_rng(0).integers(0, int(np.prod(mesh)), n).astype(np.int64)).cuda()
    H, R = torch.from_numpy(m.H_R).cuda(), np.ascontiguousarray(m.R, dtype=np.int32)
    ref = kubo.bloch(H, m.R, mesh, kidx)
    L, o = kubo.lib(), kubo.Options()
    L.kubo_options_init(ctypes.byref(o))
    o.chunk_k = chunk
    km = np.array(mesh, dtype=np.int32)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)   # noqa: E731
    size = L.kubo_workspace_size(W, m.N_R, ptr(km), 1, ctypes.byref(o))
    guard = 1 << 20
    ws = torch.full((size + guard,), 0x5A, dtype=torch.uint8, device="cuda")
    outs = [torch.empty((n, W * W), dtype=torch.float64, device="cuda") for _ in range(3)]
    o.stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    o.workspace, o.workspace_bytes = ws.data_ptr(), size
    d = lambda t: ctypes.c_void_p(t.data_ptr())   # noqa: E731
    code = L.kubo_bloch(d(H), ptr(R), W, m.N_R, ptr(km), d(kidx), n, *map(d, outs), ctypes.byref(o))
    assert code == 0
    assert bool((ws[size:] == 0x5A).all())
    col = 2.0 * np.abs(m.H_R).max() * m.N_R * half * 2.0 ** -48
    for g, r in zip(outs, ref):
        assert float((g - r).abs().max()) <= col
