"""kubo_eigh_batched: a matrix with an infinite or NaN entry has NaN eigenvalues and eigenvectors, the others theirs.

Orders around the kernels that form U (a thread per column to 16, one CTA per matrix to 64, two above).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [1, 2, 3, 8, 9, 16, 17, 32, 64, 65, 97, 128])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_matrix(W, bad):
    import torch
    import paper_2309_06675_gb300 as kubo
    rng = np.random.default_rng(W)
    z = rng.standard_normal((5, W, W)) + 1j * rng.standard_normal((5, W, W))
    P = kubo.pack_hermitian(torch.from_numpy(z + z.conj().transpose(0, 2, 1)).cuda())
    E0, U0 = kubo.eigh_batched(P, W)
    P[1, min(1, W * W - 1)] = bad   # above the diagonal
    P[3, W * W - 1] = bad           # the last diagonal entry
    E, U = kubo.eigh_batched(P, W)
    for k in (0, 2, 4):
        assert torch.equal(E[k], E0[k]) and torch.equal(U[k], U0[k])
    for k in (1, 3):
        assert torch.isnan(E[k]).all()
        assert torch.isnan(U[k].real).all() and torch.isnan(U[k].imag).all()
    only = kubo.eigh_batched(P, W, vectors=False)[0]   # by the QL iteration, as all orders up to 8
    assert torch.isnan(only[[1, 3]]).all() and torch.isfinite(only[[0, 2, 4]]).all()
