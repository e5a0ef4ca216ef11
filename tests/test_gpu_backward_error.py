"""The FP64 eigensolver's backward error: rounding of the fixed-point reduction without a bias.

U^dagger A U minus its diagonal part, (E_n + E_m) / 2 U^dagger U, is what A would have to change by for U to be
exact, in that basis.  The reduction rounds every entry W times to a unit of 2^-59 of the power of two above
the Frobenius norm: independent roundings (0.58 of a unit r.m.s. a step) leave 0.58 sqrt(W) units at most, and the
FP64 steps around them 2^-55 of the norm; a constant part of a quarter unit per step and entry leaves twice that.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [97, 112, 128])
def test_unbiased(W):
    import torch
    import paper_2309_06675_gb300 as kubo
    rng = np.random.default_rng(W)
    z = rng.standard_normal((2, W, W)) + 1j * rng.standard_normal((2, W, W))
    A = z + z.conj().transpose(0, 2, 1)
    E, U = kubo.eigh_batched(kubo.pack_hermitian(torch.from_numpy(A).cuda()), W)
    E, U = E.cpu().numpy(), U.cpu().numpy()
    for a, u in zip(A, U):
        L = np.clongdouble
        S = u.conj().T.astype(L) @ (a.astype(L) @ u.astype(L))
        G = u.conj().T.astype(L) @ u.astype(L)
        e = np.diag(S).real
        D = np.abs(S - (e[:, None] + e[None, :]) / 2 * G)[~np.eye(W, dtype=bool)]
        unit = 2.0 ** (np.ceil(np.log2(np.linalg.norm(a))) - 59)
        bound = 0.58 * np.sqrt(W) * unit + 2.0 ** -55 * np.abs(e).max()
        assert np.sqrt((D ** 2).mean()) <= bound, float(np.sqrt((D ** 2).mean()) / bound)
