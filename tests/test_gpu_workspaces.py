"""Caller's workspaces: of the queried size for every precision, and ever smaller ones where batches can shrink.

Nothing is written behind the given bytes, and the results are those of a library-managed call: the same bits
where only the batch differs, within the kernels' rounding where a smaller workspace means other kernels.
"""
import ctypes

import numpy as np
import pytest
import tbgen

pytestmark = pytest.mark.gpu
GUARD = 1 << 20


def _options(kubo, torch, size, **kw):
    o = kubo.Options()
    kubo.lib().kubo_options_init(ctypes.byref(o))
    for k, v in kw.items():
        setattr(o, k, v)
    ws = torch.full((size + GUARD,), 0x5A, dtype=torch.uint8, device="cuda")
    o.stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    o.workspace, o.workspace_bytes = ws.data_ptr(), size
    return o, ws


def _d(t):
    return ctypes.c_void_p(t.data_ptr() if t is not None else None)


@pytest.mark.parametrize("W", [3, 16, 24, 25, 64, 65, 97])
@pytest.mark.parametrize("precision", [0, 1, 2, 3, 4])
def test_queried_size(W, precision):
    import torch
    import paper_2309_06675_gb300 as kubo
    L = kubo.lib()
    m = tbgen.random_tb(W, 1, 1.5, W)
    mesh = np.array([7, 5, 4], dtype=np.int32)
    H, R = torch.from_numpy(m.H_R).cuda(), np.ascontiguousarray(m.R, dtype=np.int32)
    ef = torch.linspace(-1, 1, 3, dtype=torch.float64).cuda()
    name = {0: "fp64", 1: "mixed", 2: "mixed_fourier", 3: "mixed_rotation", 4: "mixed_df"}[precision]
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)   # noqa: E731
    for chunk, fix in ((0, 0.0), (64, 0.0), (64, 10.0 if precision in (1, 2, 4) else 0.0)):
        ref = kubo.ahc(H, m.R, tuple(mesh), ef, eta=0.05, precision=name, chunk_k=chunk, fixup_rel=fix)
        q = kubo.Options()
        L.kubo_options_init(ctypes.byref(q))
        q.precision, q.chunk_k, q.mixed_fixup_rel = precision, chunk, fix
        size = L.kubo_workspace_size(W, m.N_R, p(mesh), 3, ctypes.byref(q))
        o, ws = _options(kubo, torch, size, precision=precision, chunk_k=chunk, mixed_fixup_rel=fix)
        out = torch.zeros((1, 3), dtype=torch.float64, device="cuda")
        assert L.kubo_ahc(_d(H), p(R), W, m.N_R, p(mesh), _d(ef), 3, 0.05, _d(out), ctypes.byref(o)) == 0
        assert bool((ws[size:] == 0x5A).all())
        assert torch.equal(out, ref)


@pytest.mark.parametrize("W", [2, 8, 16, 24, 25, 33, 64, 65, 97, 128])
def test_shrinking_sizes(W):
    import torch
    import paper_2309_06675_gb300 as kubo
    L = kubo.lib()
    rng = np.random.default_rng(W)
    n = 60
    z = rng.standard_normal((3, n, W, W)) + 1j * rng.standard_normal((3, n, W, W))
    A, X, Y = (kubo.pack_hermitian(torch.from_numpy(M + M.conj().transpose(0, 2, 1)).cuda()) for M in z)
    E0, U0 = kubo.eigh_batched(A, W)
    Om0 = kubo.berry_batched(E0, U0, X, Y, eta=0.1)[0]
    norm = float(E0.abs().max())
    size, accepted = 64 << 20, {"eigh": 0, "berry": 0}
    while size >= 256:
        E, U, Om = torch.zeros_like(E0), torch.zeros_like(U0), torch.zeros_like(Om0)
        o, ws = _options(kubo, torch, size)
        code = L.kubo_eigh_batched(_d(A), W, n, _d(E), _d(U), ctypes.byref(o))
        assert code in (0, 8) and bool((ws[size:] == 0x5A).all())
        if code == 0:
            accepted["eigh"] += 1
            assert float((E - E0).abs().max()) <= 8 * W * 2.0 ** -52 * norm
            M = kubo.unpack_hermitian(A, W)
            assert float((M @ U - U * E[:, None, :]).abs().max()) <= 16 * W * 2.0 ** -52 * norm
        o, ws = _options(kubo, torch, size)
        code = L.kubo_berry_batched(_d(E0), _d(U0), _d(X), _d(Y), W, n, 0.1, _d(Om), ctypes.byref(o))
        assert code in (0, 8) and bool((ws[size:] == 0x5A).all())
        if code == 0:
            accepted["berry"] += 1
            # Omega_n: W terms of at most |v|^2 / eta^2, the velocities to 2^-50 W of their operands' norm
            big = float(kubo.unpack_hermitian(X, W).abs().max() * kubo.unpack_hermitian(Y, W).abs().max()) * W / 0.01
            assert float((Om - Om0).abs().max()) <= W * W * 2.0 ** -50 * big
        size //= 2
    assert accepted["eigh"] >= 4 and accepted["berry"] >= 6
