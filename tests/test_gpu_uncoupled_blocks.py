"""Eigensystems of matrices made of uncoupled blocks of very different scale (consecutive orbitals each).

Every block keeps the accuracy it has by itself: eigenvalues to a few roundings per step of the reduction (4 W 2^-52 of
the block's norm), eigenvectors inside the block, residuals likewise.  Without a scale per block both are off by
the ratio of the scales.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _blocks(sizes, scales, n, rng):
    W = sum(sizes)
    A = np.zeros((n, W, W), complex)
    at = 0
    for w, s in zip(sizes, scales):
        z = rng.standard_normal((n, w, w)) + 1j * rng.standard_normal((n, w, w))
        b = (z + z.conj().transpose(0, 2, 1)) / 2
        if s >= 1.0:   # the large blocks' levels away from the small ones'
            b += 100.0 * s * np.eye(w)
        A[:, at:at + w, at:at + w] = s * b
        at += w
    return A


@pytest.mark.parametrize("sizes,scales", [
    ((3, 3), (1.0, 1e-6)), ((1, 1), (1.0, 1e-9)), ((2, 1, 5), (1e-4, 1.0, 1e-8)), ((8, 8), (1e-3, 1.0)),
    ((5, 7, 5), (1.0, 1e-6, 1.0)), ((16, 16), (1.0, 1e-6)), ((1, 31, 1), (1e-6, 1.0, 1e-3)), ((32, 32), (1e-6, 1.0)),
    ((40, 25), (1.0, 1e-6)), ((48, 49), (1e-4, 1.0)), ((64, 64), (1.0, 1e-6)), ((4, 100, 24), (1e-6, 1.0, 1e-3)),
])
def test_each_block_keeps_its_accuracy(sizes, scales):
    import torch
    import paper_2309_06675_gb300 as kubo
    n, W = 5, sum(sizes)
    A = _blocks(sizes, scales, n, np.random.default_rng(W))
    A[4] = _blocks(sizes, [1.0] * len(sizes), 1, np.random.default_rng(1))[0]   # one of a single scale beside them
    E, U = kubo.eigh_batched(kubo.pack_hermitian(torch.from_numpy(A).cuda()), W)
    only = kubo.eigh_batched(kubo.pack_hermitian(torch.from_numpy(A).cuda()), W, vectors=False)[0].cpu().numpy()
    E, U = E.cpu().numpy(), U.cpu().numpy()
    L = np.clongdouble
    for k in range(4):
        at = 0
        for w, s in zip(sizes, scales):
            ref = np.linalg.eigvalsh(A[k, at:at + w, at:at + w])
            norm = np.abs(ref).max()
            inside = (np.abs(U[k, at:at + w]) ** 2).sum(0)
            if s < 1.0:
                m = np.flatnonzero(inside > 0.5)
                assert len(m) == w
                assert np.abs(E[k, m] - ref).max() <= 4 * W * 2.0 ** -52 * norm
                near = np.abs(only[k][:, None] - ref[None]).min(0)
                assert near.max() <= 4 * W * 2.0 ** -52 * norm
                u = U[k][:, m].astype(L)
                assert np.abs(A[k].astype(L) @ u - u * E[k, m]).max() <= 8 * W * 2.0 ** -52 * norm
            at += w
        G = U[k].conj().T.astype(L) @ U[k].astype(L)
        assert np.abs(G - np.eye(W)).max() <= 8 * W * 2.0 ** -52
    ref = np.linalg.eigvalsh(A[4])
    assert np.abs(E[4] - ref).max() <= 4 * W * 2.0 ** -52 * np.abs(ref).max()
