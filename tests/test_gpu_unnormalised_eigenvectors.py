"""kubo_berry_batched with eigenvectors whose norms differ a little from a power of two.

The products' operands are scaled by powers of two: a dominating diagonal entry just below its power and
columns just above theirs leave the least room.  Bound: v to 2^-49 W of its largest entry (test_gpu_fixed.py).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _near_identity(W, rng):
    G = rng.standard_normal((W, W)) + 1j * rng.standard_normal((W, W))
    K = 1e-3 * (G - G.conj().T)
    return np.linalg.qr(np.eye(W) + K)[0]


@pytest.mark.parametrize("W", [2, 3, 12, 13, 24, 25, 33, 65])
@pytest.mark.parametrize("norm", [1.0 + 2.0 ** -40, 1.0 + 2.0 ** -33, 1.0009, 1.0 - 2.0 ** -12, 2.0009, 0.50001])
@pytest.mark.parametrize("top", [0.9995, 1.0 - 2.0 ** -16, 1.0 - 2.0 ** -52, 1.0])
def test_norms_at_the_edge(W, norm, top):
    import torch
    import paper_2309_06675_gb300 as kubo
    rng = np.random.default_rng(W)
    n = 3
    U = np.stack([_near_identity(W, rng) for _ in range(n)]) * norm
    X, Y = (np.zeros((n, W, W), complex) for _ in range(2))
    for A in (X, Y):
        z = 1e-3 * (rng.standard_normal((n, W, W)) + 1j * rng.standard_normal((n, W, W)))
        A += z + z.conj().transpose(0, 2, 1)
    X[:, W - 1, W - 1] = top
    Y[:, 0, 0] = -top
    E = np.sort(rng.standard_normal((n, W)), axis=1)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    got = kubo.berry_batched(d(E), d(U), kubo.pack_hermitian(d(X)), kubo.pack_hermitian(d(Y)),
                             eta=0.3).cpu().numpy()[0]
    L = np.clongdouble
    Uh = U.conj().transpose(0, 2, 1).astype(L)
    vx, vy = (Uh @ A.astype(L) @ U.astype(L) for A in (X, Y))
    d2 = (E[:, :, None] - E[:, None, :]).astype(np.longdouble) ** 2 + np.longdouble(0.3) ** 2
    T = -2 * (vx * vy.conj()).imag / d2
    T[:, np.arange(W), np.arange(W)] = 0
    size = (np.abs(vx).max((1, 2)) * np.abs(vy).max((1, 2)))[:, None, None] / d2
    bound = (size * W * 2.0 ** -49).sum(2)
    assert (np.abs(got - T.sum(2)) <= bound).all(), float((np.abs(got - T.sum(2)) / bound).max())
