"""The k-sum at a temperature for kT from 10^-12 to 10^2 of the band energies.

Levels and Fermi levels of the same sign far from zero (|E| / kT up to 10^13), Fermi levels on, beside and between
levels, and infinite ones.  Reference: the occupations of the same levels in extended precision.  A pair's
occupation f is a few roundings, or carries the rounding of x = (E - E_F) / kT (f (1 - f) |x| 2^-52); the
sum adds one rounding per term.
"""
import numpy as np
import pytest
import tbgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kT", [1e-12, 1e-10, 1e-9, 1e-8, 2.4e-8, 2.7e-8, 8.6e-8, 1e-6, 1e-3, 1.0, 1e2])
@pytest.mark.parametrize("shift", [9.0, -9.0, 0.0])
@pytest.mark.parametrize("n_EF", [1, 12, 300])
def test_occupations(kT, shift, n_EF):
    import torch
    import paper_2309_06675_gb300 as kubo
    W, mesh, etas = 6, (5, 3, 4), [0.05, 0.3]
    m = tbgen.random_tb(W, 1, 1.0, 4)
    H = m.H_R.copy()
    H[np.flatnonzero((m.R == 0).all(1))[0]] += shift * np.eye(W)
    Hd, R = torch.from_numpy(H).cuda(), m.R
    n = int(np.prod(mesh))
    E, Om = kubo.ahc_k(Hd, R, mesh, torch.arange(n, dtype=torch.int64).cuda(), etas=etas)
    E, Om = E.cpu().numpy(), Om.cpu().numpy()
    lev = np.sort(E.ravel())
    rng = np.random.default_rng(1)
    near = lev[rng.integers(0, lev.size, 300)] + kT * rng.choice([0.0, 0.3, -2.0, 30.0, -700.0], 300)
    ef = np.concatenate([[np.inf, -np.inf, lev[0] - 1.0, lev[-1] + 1.0, 0.5 * (lev[10] + lev[11]), 0.0], near])
    ef = ef[:n_EF] if n_EF > 1 else ef[6:7]
    got = kubo.ahc(Hd, R, mesh, torch.from_numpy(ef).cuda(), etas=etas, kT=kT).cpu().numpy()
    L = np.longdouble
    x = (E[None].astype(L) - ef[:, None, None].astype(L)) / L(kT)
    ex = np.exp(-np.minimum(np.abs(x), 11000))
    f = np.where(x > 0, ex / (1 + ex), 1 / (1 + ex))
    df = f * (L(2.0) ** -48 + np.minimum(np.abs(x), 11000) * np.minimum(1, ex) * L(2.0) ** -50) + L(2.0) ** -990
    df += f * (f < 0.5) * np.minimum(np.abs(x), 11000) * L(2.0) ** -50
    for e in range(2):
        ref = (f * Om[e].astype(L)).sum((1, 2)) / n
        bound = (df * np.abs(Om[e])).sum((1, 2)) / n + (W + 4) * 2.0 ** -52 * (f * np.abs(Om[e])).sum((1, 2)) / n
        assert (np.abs(got[e] - ref) <= bound).all(), float((np.abs(got[e] - ref) / bound).max())
