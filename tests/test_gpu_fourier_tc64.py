"""FP64 Fourier sum on the tensor cores (seven slices) against an extended-precision sum.

Sizes around its tiles: 32 columns (3 W^2 mod 32), 128 k-points, 64 of K (N_R), one or several
drain groups, sub-batches of one row.  Bound per entry: phases of three FP64 factors (2^-51 each),
operand rounding (2 x 2^-56) and dropped levels (6.1 x 2^-56) on N_R terms of at most the column's
largest basis entry (A_h and B_h add two blocks: twice the largest |H(R)|, times |R_a|).
"""
import numpy as np
import pytest
import tbgen

pytestmark = pytest.mark.gpu


def _reference(m, kmesh, kidx):
    N = np.array(kmesh)
    j = np.stack([kidx // (N[1] * N[2]), (kidx // N[2]) % N[1], kidx % N[2]], 1)
    turn = np.zeros((len(kidx), m.N_R), dtype=np.longdouble)
    for a in range(3):
        turn += ((j[:, a:a + 1] * m.R[None, :, a].astype(np.int64)) % N[a]).astype(np.longdouble) / N[a]
    pi = np.longdouble("3.14159265358979323846264338327950288")
    ph = np.cos(2 * pi * turn) + 1j * np.sin(2 * pi * turn)
    flat = m.H_R.reshape(m.N_R, -1).astype(np.clongdouble)
    w = [np.ones(m.N_R), 1j * m.R[:, 0], 1j * m.R[:, 1]]
    return [((ph * x[None]) @ flat).reshape(-1, m.W, m.W) for x in w]


@pytest.mark.parametrize("W,half,kmesh,n", [
    (5, 5, (31, 17, 9), 4500),     # 75 columns: odd W^2, padding columns, 36 row tiles
    (33, 1, (7, 6, 5), 800),       # 3267 columns, one K block (27 vectors)
    (24, 2, (40, 3, 11), 129),     # 125 vectors: two K blocks, one row in the second tile
    (64, 3, (64, 64, 64), 1),      # a single row
    (97, 2, (9, 9, 9), 127),
])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 60])
def test_matches_extended_precision(W, half, kmesh, n, scale):
    import torch
    import paper_2309_06675_gb300 as kubo
    m = tbgen.random_tb(W, half, 1.5, seed=W)
    m = tbgen.TBModel(H_R=m.H_R * scale, R=m.R)
    rng = np.random.default_rng(3)
    kidx = rng.integers(0, int(np.prod(kmesh)), n).astype(np.int64)
    got = kubo.bloch(torch.from_numpy(m.H_R).cuda(), m.R, kmesh, torch.from_numpy(kidx).cuda())
    probe = np.unique(np.concatenate([np.arange(min(n, 6)), np.arange(max(0, n - 6), n)]))
    ref = _reference(m, kmesh, kidx[probe])
    col = 2.0 * np.abs(m.H_R).max(axis=0)
    for a, (g, r) in enumerate(zip(got, ref)):
        A = kubo.unpack_hermitian(g[torch.from_numpy(probe).cuda()], W).cpu().numpy()
        big = 1.0 if a == 0 else float(half)
        bound = m.N_R * np.maximum(col, col.T) * big * (3 * 2.0 ** -51 + 8.1 * 2.0 ** -56)
        assert (np.abs(A - r) <= bound[None]).all(), float((np.abs(A - r) / bound[None]).max())
