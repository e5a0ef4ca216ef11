"""Step (1) in FP64 for few k-points, on both sides of the line between its two kernels (orders, vectors, k-points).

Bound: N_R terms of a column's largest basis entry, each 2^-48 (the FP64-pipe chain's).
"""
import numpy as np
import pytest
import tbgen

from test_gpu_long_ranges import _reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [4, 64, 80, 91, 128])
@pytest.mark.parametrize("half", [1, 2])
@pytest.mark.parametrize("n", [1, 16, 17, 32, 33, 128, 129])
def test_few_k_points(W, half, n):
    import torch
    import paper_2309_06675_gb300 as kubo
    m = tbgen.random_tb(W, half, 1.5, seed=W)
    mesh = (13, 9, 7)
    kidx = np.random.default_rng(n).integers(0, int(np.prod(mesh)), n).astype(np.int64)
    got = kubo.bloch(torch.from_numpy(m.H_R).cuda(), m.R, mesh, torch.from_numpy(kidx).cuda())
    probe = np.unique([0, n // 2, n - 1])
    ref = _reference(m.H_R, m.R, mesh, kidx[probe])
    col = 2.0 * np.abs(m.H_R).max(axis=0)
    col = np.maximum(col, col.T) * m.N_R * half * 2.0 ** -48
    for g, r in zip(got, ref):
        A = kubo.unpack_hermitian(g[torch.from_numpy(probe).cuda()], W).cpu().numpy()
        assert (np.abs(A - r) <= col[None]).all()
