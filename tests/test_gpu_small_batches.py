"""kubo_berry_batched below and above the batch size at which its small-order kernel changes (1,216 matrices, W <= 16).

The velocities are the same fixed-point sums either way; a band's sum over its W - 1 pairs is grouped otherwise.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [1, 2, 5, 6, 12, 13, 15, 16, 17])
def test_few_and_many(W):
    import torch
    import paper_2309_06675_gb300 as kubo
    rng = np.random.default_rng(W)
    n = 1217
    z = rng.standard_normal((3, n, W, W)) + 1j * rng.standard_normal((3, n, W, W))
    A = z + z.conj().transpose(0, 1, 3, 2)
    E, U = np.linalg.eigh(A[0])
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    E, U, X, Y = d(E), d(U), kubo.pack_hermitian(d(A[1])), kubo.pack_hermitian(d(A[2]))
    etas = [0.0, 1e-2, 0.5]
    whole = kubo.berry_batched(E, U, X, Y, etas=etas).cpu().numpy()
    for a, b in ((0, 1216), (0, 1), (1210, 1217), (300, 1001)):
        part = kubo.berry_batched(E[a:b], U[a:b], X[a:b], Y[a:b], etas=etas).cpu().numpy()
        dE = E[a:b, :, None].cpu().numpy() - E[a:b, None, :].cpu().numpy()
        vx, vy = (np.abs((U[a:b].mH @ kubo.unpack_hermitian(M[a:b], W) @ U[a:b]).cpu().numpy()) for M in (X, Y))
        for e, eta in enumerate(etas):
            den = dE ** 2 + eta ** 2 + (dE == 0)
            size = (2.0 * vx * vy / den).sum(2)
            assert (np.abs(part[e] - whole[e, a:b]) <= (W + 4) * 2.0 ** -51 * size).all()
