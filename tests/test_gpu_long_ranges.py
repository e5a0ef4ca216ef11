"""Step (1) where its index arithmetic leaves 32 bits: many rows of many vectors, long mesh axes.

Bounds as in test_gpu_fourier_tc64.py (FP64 mode); the mixed form's is 2^-29 of the sum of magnitudes
(operands to 31 fractional bits, phases to 2^-44).
"""
import numpy as np
import pytest
import tbgen

pytestmark = pytest.mark.gpu


def _reference(H, R, kmesh, kidx):
    N = np.array(kmesh, dtype=np.int64)
    j = np.stack([kidx // (N[1] * N[2]), (kidx // N[2]) % N[1], kidx % N[2]], 1)
    turn = np.zeros((len(kidx), len(R)), dtype=np.longdouble)
    for a in range(3):
        turn += ((j[:, a:a + 1] * R[None, :, a].astype(np.int64)) % N[a]).astype(np.longdouble) / N[a]
    pi = np.longdouble("3.14159265358979323846264338327950288")
    ph = np.cos(2 * pi * turn) + 1j * np.sin(2 * pi * turn)
    flat = H.reshape(len(R), -1).astype(np.clongdouble)
    w = [np.ones(len(R)), 1j * R[:, 0], 1j * R[:, 1]]
    return [((ph * x[None]) @ flat).reshape(-1, H.shape[1], H.shape[1]) for x in w]


def _check(H, R, kmesh, kidx, probe, precision):
    import torch
    import paper_2309_06675_gb300 as kubo
    W = H.shape[1]
    got = kubo.bloch(torch.from_numpy(H).cuda(), R, kmesh, torch.from_numpy(kidx).cuda(), precision=precision)
    ref = _reference(H, R, kmesh, kidx[probe])
    col = 2.0 * np.abs(H).max(axis=0)
    col = np.maximum(col, col.T)
    each = 3 * 2.0 ** -51 + 8.1 * 2.0 ** -56 if precision == "fp64" else 2.0 ** -29
    for a, (g, r) in enumerate(zip(got, ref)):
        A = kubo.unpack_hermitian(g[torch.from_numpy(probe).cuda()], W).cpu().numpy()
        big = 1.0 if a == 0 else float(np.abs(R[:, a - 1]).max())
        bound = len(R) * col * big * each
        assert (np.abs(A - r) <= bound[None]).all(), (a, float((np.abs(A - r) / bound[None]).max()))


@pytest.mark.parametrize("N_R,rows", [(1343, 40_000), (959, 45_000)])   # N_R = 63 mod 64: the last pair is R = 0
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_many_rows(N_R, rows, precision):
    m = tbgen.random_tb(4, 6, 2.0, seed=1)
    order = np.argsort((m.R.astype(np.int64) ** 2).sum(1), kind="stable")
    pick, seen = [], set()
    for i in order:   # the N_R shortest vectors with their negatives
        if tuple(m.R[i]) in seen:
            continue
        pair = {tuple(m.R[i]), tuple(-m.R[i])}
        if len(seen) + len(pair) > N_R:
            break
        seen |= pair
    keep = np.array([tuple(r) in seen for r in m.R])
    H, R = np.ascontiguousarray(m.H_R[keep]), np.ascontiguousarray(m.R[keep])
    assert len(R) == N_R
    kmesh = (61, 53, 47)
    kidx = np.random.default_rng(0).integers(0, int(np.prod(kmesh)), rows).astype(np.int64)
    probe = np.concatenate([np.arange(4), np.arange(rows // 2, rows // 2 + 8), np.arange(rows - 40, rows)])
    _check(H, R, kmesh, kidx, probe, precision)


@pytest.mark.parametrize("kmesh", [(90001, 1, 1), (2, 90001, 1), (3, 2, 1000003)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_long_axes(kmesh, precision):
    m = tbgen.random_tb(5, 2, 1.5, seed=2)
    n = int(np.prod(np.array(kmesh, dtype=np.int64)))
    kidx = np.concatenate([np.arange(32), np.arange(n - 96, n)]).astype(np.int64)
    _check(m.H_R, m.R, kmesh, kidx, np.arange(len(kidx)), precision)
