"""Integer-pipe products of FP64 grade (rotations, U = Q D Z) against extended precision.

Orders around the tiles (2 x 2 below 13, 4 x 2 to 24, tensor-core tiles of up to 64 above; 4 reflectors
per block), magnitudes far from
1, eigenvectors that are not normalised, non-finite operands.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(W, n, seed):
    rng = np.random.default_rng(seed)
    z = rng.standard_normal((3, n, W, W)) + 1j * rng.standard_normal((3, n, W, W))
    A = z + z.conj().transpose(0, 1, 3, 2)
    E, U = np.linalg.eigh(A[0])
    return A, E, U


def _velocities(U, X, Y):
    L = np.clongdouble
    Uh = U.conj().transpose(0, 2, 1).astype(L)
    return Uh @ X.astype(L) @ U.astype(L), Uh @ Y.astype(L) @ U.astype(L)


def _curvature(E, vx, vy, eta):
    d2 = (E[:, :, None] - E[:, None, :]).astype(np.longdouble) ** 2 + np.longdouble(eta) ** 2
    num = -2 * (vx * vy.conj()).imag
    T = num / np.where(d2 == 0, 1, d2)
    T[:, np.arange(E.shape[1]), np.arange(E.shape[1])] = 0
    # size of the terms that enter Omega_n, for the error bound
    size = (np.abs(vx).max((1, 2)) * np.abs(vy).max((1, 2)))[:, None, None] / d2
    return T.sum(2), size


@pytest.mark.parametrize("W", [1, 2, 3, 4, 5, 11, 12, 13, 16, 24, 25, 32, 33, 48, 63, 64, 65, 97, 128])
@pytest.mark.parametrize("sx,sy,su", [(1.0, 1.0, 1.0), (2.0 ** 130, 2.0 ** -90, 1.0), (1.0, 1.0, 3.0)])
def test_curvature(W, sx, sy, su):
    import torch
    import paper_2309_06675_gb300 as kubo
    n = 7 if W <= 64 else 2
    A, E, U = _problem(W, n, W)
    X, Y, U = A[1] * sx, A[2] * sy, U * su
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    got = kubo.berry_batched(d(E), d(U), kubo.pack_hermitian(d(X)), kubo.pack_hermitian(d(Y)),
                             etas=[1e-2, 0.5]).cpu().numpy()
    vx, vy = _velocities(U, X, Y)
    for e, eta in enumerate([1e-2, 0.5]):
        ref, size = _curvature(E, vx, vy, eta)
        # v to 2^-51 of the norm of the operands (at most W times the largest entry of v)
        bound = (size * W * 2.0 ** -49).sum(2)
        assert (np.abs(got[e] - ref) <= bound).all(), float((np.abs(got[e] - ref) / bound).max())


def test_non_finite_operands():
    import torch
    import paper_2309_06675_gb300 as kubo
    A, E, U = _problem(20, 4, 1)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    X = kubo.pack_hermitian(d(A[1]))
    Y = kubo.pack_hermitian(d(A[2]))
    X[1, 7] = float("inf")
    Ud = d(U)
    Ud[2, 3, 4] = float("nan")
    got = kubo.berry_batched(d(E), Ud, X, Y, eta=0.1).cpu().numpy()[0]
    assert np.isfinite(got[0]).all() and np.isfinite(got[3]).all()
    assert np.isnan(got[1]).all() and np.isnan(got[2]).all()


@pytest.mark.parametrize("W", [1, 2, 3, 6, 7, 18, 32, 33, 47, 64])
def test_eigenvectors(W):
    import torch
    import paper_2309_06675_gb300 as kubo
    n = 9
    A = _problem(W, n, 100 + W)[0][0]
    E, U = kubo.eigh_batched(kubo.pack_hermitian(torch.from_numpy(A).cuda()), W)
    E, U = E.cpu().numpy(), U.cpu().numpy()
    L = np.clongdouble
    norm = np.abs(E).max(1)[:, None, None]
    res = np.abs(A.astype(L) @ U.astype(L) - U.astype(L) * E[:, None, :]) / norm
    orth = np.abs(U.conj().transpose(0, 2, 1).astype(L) @ U.astype(L) - np.eye(W))
    # a W-step reduction at 2^-52 of the norm per step and entry
    assert res.max() <= 4 * W * 2.0 ** -52 and orth.max() <= 4 * W * 2.0 ** -52, (res.max(), orth.max())


def _structured(kind, W, n, rng):
    """Matrices whose spectra are hard for shifts: exact and near multiples, splits, one scale apart."""
    z = rng.standard_normal((n, W, W)) + 1j * rng.standard_normal((n, W, W))
    Q = np.linalg.qr(z)[0]
    lam = rng.standard_normal((n, W))
    if kind == "pairs":
        lam[:, 1::2] = lam[:, : 2 * (W // 2): 2]
    elif kind == "close":
        lam[:, 1::2] = lam[:, : 2 * (W // 2): 2] + 10.0 ** rng.uniform(-15, -4, (n, W // 2))
    elif kind == "one":
        lam[:] = 0.75
    elif kind == "graded":
        lam *= 2.0 ** -np.linspace(0, 40, W)
    A = (Q * lam[:, None, :]) @ Q.conj().transpose(0, 2, 1)
    if kind == "blocks":
        A[:, : W // 2, W // 2:] = 0
        A[:, W // 2:, : W // 2] = 0
    if kind == "diagonal":
        A = np.stack([np.diag(x) for x in lam]).astype(complex)
    if kind == "zero":
        A[:] = 0
    return (A + A.conj().transpose(0, 2, 1)) / 2


@pytest.mark.parametrize("W", [9, 10, 33, 64, 65, 128])
@pytest.mark.parametrize("kind", ["pairs", "close", "one", "graded", "blocks", "diagonal", "zero"])
def test_eigensystem_of_structured_matrices(W, kind):
    import torch
    import paper_2309_06675_gb300 as kubo
    A = _structured(kind, W, 5, np.random.default_rng(W))
    E, U = kubo.eigh_batched(kubo.pack_hermitian(torch.from_numpy(A).cuda()), W)
    E, U = E.cpu().numpy(), U.cpu().numpy()
    ref = np.linalg.eigvalsh(A)
    norm = max(np.abs(ref).max(), 1e-300)
    assert (np.diff(E, axis=1) >= 0).all()
    assert np.abs(E - ref).max() <= 4 * W * 2.0 ** -52 * norm
    assert np.abs(A @ U - U * E[:, None, :]).max() <= 8 * W * 2.0 ** -52 * norm
    assert np.abs(U.conj().transpose(0, 2, 1) @ U - np.eye(W)).max() <= 8 * W * 2.0 ** -52


def test_non_finite_matrix_leaves_the_others():
    import torch
    import paper_2309_06675_gb300 as kubo
    A = _structured("pairs", 20, 3, np.random.default_rng(0))
    P = kubo.pack_hermitian(torch.from_numpy(A).cuda())
    P[1, 5] = float("nan")
    E = kubo.eigh_batched(P, 20)[0].cpu().numpy()
    ref = np.linalg.eigvalsh(A)
    assert np.isnan(E[1]).all()
    assert np.abs(E[[0, 2]] - ref[[0, 2]]).max() <= 80 * 2.0 ** -52 * np.abs(ref).max()


def test_non_finite_operands_in_a_shared_tile():
    # two matrices of order 25 .. 32 to a tensor-core tile: the other one is not affected
    import torch
    import paper_2309_06675_gb300 as kubo
    A, E, U = _problem(30, 5, 2)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    X = kubo.pack_hermitian(d(A[1]))
    Y = kubo.pack_hermitian(d(A[2]))
    ref = kubo.berry_batched(d(E), d(U), X, Y, eta=0.1).cpu().numpy()[0]
    X[1, 7] = float("inf")
    Ud = d(U)
    Ud[2, 3, 4] = float("nan")
    got = kubo.berry_batched(d(E), Ud, X, Y, eta=0.1).cpu().numpy()[0]
    assert np.array_equal(got[[0, 3, 4]], ref[[0, 3, 4]])
    assert np.isnan(got[1]).all() and np.isnan(got[2]).all()


@pytest.mark.parametrize("W", [1, 5, 15, 16, 17, 31, 32, 33])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 6])
def test_gradient_of_shared_tiles(W, n):
    # Four (W <= 16) or two (W <= 32) k-points share a tile of the gradient's products, one by itself
    # when the range is a single k-point.  The products of a k-point are the same numbers either way;
    # the sum over k rounds its operands to 2^-55 of the largest of the range.
    import torch
    import tbgen
    import paper_2309_06675_gb300 as kubo
    m = tbgen.random_tb(W, 1, 1.0, W)
    H, R = torch.from_numpy(m.H_R).cuda(), torch.from_numpy(m.R)
    E_F = torch.zeros(1, dtype=torch.float64, device="cuda")
    g = torch.ones(1, 1, dtype=torch.float64, device="cuda")
    run = lambda a, b: kubo.ahc_grad(H, R, (4, 3, 2), E_F, g, etas=[0.05], kT=0.1, k_range=(a, b))   # noqa: E731
    first = lambda x: x[0] if isinstance(x, tuple) else x   # noqa: E731
    whole = first(run(3, 3 + n)).cpu().numpy()
    parts = sum(first(run(3 + i, 4 + i)).cpu().numpy() for i in range(n))
    assert np.isfinite(whole).all()
    assert np.abs(whole - parts).max() <= 1e-12 * max(np.abs(parts).max(), 1e-300)


@pytest.mark.parametrize("n_EF", [1, 2, 3, 31, 33, 255, 256, 257])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 70])
def test_step_occupation_sum(n_EF, n):
    # Fermi levels x groups of k-points of a block (32 k-points): against an exact sum of the same
    # curvatures; a compensated sum of at most 70 terms of one rounding each (the prefix over bands: W of them)
    import math
    import torch
    import tbgen
    import paper_2309_06675_gb300 as kubo
    W, mesh, etas = 5, (5, 7, 2), [0.05, 0.3]
    m = tbgen.random_tb(W, 1, 1.0, 3)
    H, R = torch.from_numpy(m.H_R).cuda(), torch.from_numpy(m.R)
    ef = np.linspace(-1.5, 1.5, n_EF)
    got = kubo.ahc(H, R, mesh, torch.from_numpy(ef).cuda(), etas=etas, k_range=(0, n)).cpu().numpy()
    E, Om = kubo.ahc_k(H, R, mesh, torch.arange(n, dtype=torch.int64).cuda(), etas=etas)
    E, Om = E.cpu().numpy(), Om.cpu().numpy()
    for e in range(2):
        for j in range(n_EF):
            occ = E < ef[j]
            ref = math.fsum(Om[e][occ]) / np.prod(mesh)
            bound = (W + 2) * 2.0 ** -52 * np.abs(Om[e][occ]).sum() / np.prod(mesh)
            assert abs(got[e, j] - ref) <= bound, (e, j)
