"""The calls whose speed is measured: what programs built on this library ask of it.

A case names a kind of call (the public entry point it goes through) and its sizes; `prepare` makes
what the calling program has in hand (the model, the mesh, the Fermi levels), `run` makes the one
call, `exact` evaluates the same formulas in plain 64-bit torch.  Models are random Hermitian-paired
tight-binding models with decaying hoppings, a N(0,1) exp(i phi) exp(-|R| / 1.5), whose random phases
break time reversal, and stacks of the two-band Haldane model.
"""
import math

import numpy as np
import torch

import paper_2309_06675_gb300 as kubo

DECAY = 1.5
ETA_SWEEP = (1e-3, 1e-4, 5e-3, 1e-2)   # broadenings of a sweep, the first one alone otherwise


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # Quantised conductance of a small stacked two-band model on a fine 2-D mesh, with every
        # broadening of the sweep: tiny matrices, very many of them.
        dict(name="ahc_haldane_384x384", kind="ahc", model="haldane", W=6, half=1, n1=384, n2=384, n3=1,
             k0=0, nk=147456, n_ef=1, n_eta=4, kT=0.0, precision="fp64"),
        # The smallest call: a two-band model on a coarse mesh, inside a loop over parameters on
        # the host (buffers in host memory).
        dict(name="ahc_host_two_band", kind="ahc_host", model="haldane", W=2, half=1, n1=24, n2=24, n3=1,
             k0=0, nk=576, n_ef=1, n_eta=1, kT=0.0, precision="fp64"),
        # The plain calculation: one material of 16 orbitals, 24^3 mesh, one Fermi level.
        dict(name="ahc_w16_24cubed", kind="ahc", model="random", W=16, half=2, n1=24, n2=24, n3=24,
             k0=0, nk=13824, n_ef=1, n_eta=1, kT=0.0, precision="fp64"),
        # A 64-orbital cell with long-range hoppings, 64 Fermi levels: a quarter of a k1-plane of the
        # 128^3 mesh in full precision ...
        dict(name="ahc_w64_fp64", kind="ahc", model="random", W=64, half=5, n1=128, n2=128, n3=128,
             k0=16384, nk=4096, n_ef=64, n_eta=1, kT=0.0, precision="fp64"),
        # ... and four planes of it in the mixed-precision form.
        dict(name="ahc_w64_mixed", kind="ahc", model="random", W=64, half=5, n1=128, n2=128, n3=128,
             k0=65536, nk=65536, n_ef=64, n_eta=1, kT=0.0, precision="mixed"),
        # Supercell of the largest order, 512 Fermi levels and four broadenings, mixed precision.
        dict(name="sweep_w128_mixed", kind="ahc", model="random", W=128, half=5, n1=96, n2=96, n3=96,
             k0=9216, nk=9216, n_ef=512, n_eta=4, kT=0.0, precision="mixed"),
        # A supercell of an odd order above 64 in full precision.
        dict(name="ahc_w97_fp64", kind="ahc", model="random", W=97, half=3, n1=14, n2=14, n3=14,
             k0=0, nk=2744, n_ef=5, n_eta=1, kT=0.0, precision="fp64"),
        # Conductivity against the chemical potential at a temperature: 201 levels, two broadenings.
        dict(name="ahc_w32_thermal", kind="ahc", model="random", W=32, half=4, n1=48, n2=48, n3=48,
             k0=0, nk=4608, n_ef=201, n_eta=2, kT=0.025, precision="fp64"),
        # Many materials of uneven sizes in one call (high-throughput screening).
        dict(name="batched_8_models", kind="batched", models=8, w_lo=8, w_hi=96, half_lo=3, half_hi=5,
             n_lo=12, n_hi=24, shapes=7, precision="mixed"),
        # Fitting a model: the conductivity and its gradient with respect to every hopping.
        dict(name="grad_w32", kind="grad", model="random", W=32, half=4, n1=48, n2=48, n3=48,
             k0=0, nk=9216, n_ef=1, n_eta=1, kT=0.025, precision="fp64"),
        # Band energies and curvatures along a path of listed k-points, an odd number of them.
        dict(name="bands_w48_777", kind="ahc_k", model="random", W=48, half=3, n1=60, n2=60, n3=60,
             nk=777, n_eta=1, precision="fp64"),
        # The steps one by one: Bloch matrices, their eigensystems, the curvatures from them.
        dict(name="steps_w24_3001", kind="steps", model="random", W=24, half=3, n1=40, n2=40, n3=40,
             nk=3001, n_eta=2, precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fp64_flops(W, N_R):
    """Operations of one k-point: Fourier sum over the Hermitian half set, eigensystem, rotations."""
    return 6.0 * N_R * W * W + (16.0 / 3.0 + 8.0 + 24.0) * W ** 3


def draw(rng):
    kind = rng.choice(["ahc", "ahc", "ahc", "ahc_host", "ahc_k", "steps", "grad", "batched"])
    if kind == "batched":
        n_lo = rng.randint(8, 16)
        return dict(kind=kind, models=rng.randint(2, 8), w_lo=8, w_hi=rng.randint(24, 96), half_lo=2,
                    half_hi=rng.randint(3, 5), n_lo=n_lo, n_hi=n_lo + rng.randint(0, 8),
                    shapes=rng.randint(100, 999), precision=rng.choice(["mixed", "fp64"]))
    W = _log_int(rng, 2, 64 if kind == "grad" else 128)
    half = rng.randint(1, 5)
    precision = rng.choice(["fp64", "fp64", "mixed"]) if kind == "ahc" else "fp64"
    n1, n2, n3 = rng.randint(20, 96), rng.randint(20, 96), rng.randint(1, 64)
    # k-points: over the whole range that a third of a second of full-precision arithmetic allows
    # (the gradient counts three times)
    per_k = _fp64_flops(W, (2 * half + 1) ** 3) * (3.0 if kind == "grad" else 1.0) + 2e4
    most = max(64, min(n1 * n2 * n3, 65536, int(3e11 / per_k)))
    nk = min(n1 * n2 * n3, _log_int(rng, 64, most))
    c = dict(kind=kind, model="random", W=W, half=half, n1=n1, n2=n2, n3=n3, nk=nk,
             n_eta=rng.choice([1, 1, 2, 4]), precision=precision)
    if kind in ("ahc", "ahc_host", "grad"):
        c.update(k0=rng.randint(0, n1 * n2 * n3 - nk), n_ef=_log_int(rng, 1, 16 if kind == "grad" else 512),
                 kT=rng.choice([0.0, 0.025]) if kind != "grad" else 0.025)
    return c


# --------------------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (int(seed) + 1))
    return g


def _box(half):
    ax = np.arange(-half, half + 1, dtype=np.int32)
    return np.ascontiguousarray(np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3))


def _random_model(W, half, g):
    """H(R) on the box {-half..half}^3 (lexicographic order, so -R is at N_R - 1 - i)."""
    R = _box(half)
    n = R.shape[0]
    f = dict(dtype=torch.float64, device="cuda", generator=g)
    a = torch.randn((n, W, W), **f)
    phi = 2.0 * math.pi * torch.rand((n, W, W), **f)
    scale = torch.from_numpy(np.exp(-np.linalg.norm(R, axis=1) / DECAY)).cuda()
    H = torch.polar(torch.ones_like(a), phi) * (a * scale[:, None, None])
    mid = n // 2
    H[:mid] = H[mid + 1:].flip(0).conj().transpose(1, 2)
    H0 = torch.triu(H[mid], 1)
    H[mid] = H0 + H0.conj().T + torch.diag(torch.diagonal(a[mid]).to(H.dtype))
    return H.contiguous(), R


def _haldane_model(W, g):
    """W / 2 uncoupled Haldane layers in their topological phase, couplings drawn per call."""
    u = torch.rand(3, dtype=torch.float64, device="cuda", generator=g).tolist()
    t1, t2, phi, M = 1.0, 0.08 + 0.08 * u[0], math.pi * (0.4 + 0.2 * u[1]), 0.1 * (u[2] - 0.5)
    acc = {}

    def hop(r, i, j, v):
        for rr, ii, jj, vv in ((r, i, j, v), (tuple(-x for x in r), j, i, np.conj(v))):
            acc.setdefault(rr, np.zeros((2, 2), dtype=np.complex128))[ii, jj] += vv

    acc[(0, 0, 0)] = np.diag([M, -M]).astype(np.complex128)
    for r in [(0, 0, 0), (-1, 0, 0), (0, -1, 0)]:
        hop(r, 0, 1, t1)
    for r in [(1, 0, 0), (-1, 1, 0), (0, -1, 0)]:
        hop(r, 0, 0, t2 * np.exp(1j * phi))
        hop(r, 1, 1, t2 * np.exp(-1j * phi))
    keys = sorted(acc)
    H = np.stack([np.kron(np.eye(W // 2), acc[k]) for k in keys])
    return torch.from_numpy(np.ascontiguousarray(H)).cuda(), np.array(keys, dtype=np.int32)


def _model(c, g):
    return _haldane_model(c["W"], g) if c["model"] == "haldane" else _random_model(c["W"], c["half"], g)


def _fermi(c, g):
    """Fermi levels: in the gap of the Haldane model, a grid over the middle of the bands otherwise."""
    off = float(torch.rand(1, dtype=torch.float64, device="cuda", generator=g))
    n = c["n_ef"]
    if c["model"] == "haldane":
        return torch.full((n,), 0.02 * (off - 0.5), dtype=torch.float64, device="cuda")
    if n == 1:
        return torch.tensor([off - 0.5], dtype=torch.float64, device="cuda")
    return torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device="cuda") + 0.01 * off


def _etas(c):
    return list(ETA_SWEEP[:c["n_eta"]])


def _shapes(c):
    """The uneven models of a batch: (W, half, N) from the case alone."""
    r = np.random.default_rng(c["shapes"])
    return [(int(r.integers(c["w_lo"], c["w_hi"] + 1)), int(r.integers(c["half_lo"], c["half_hi"] + 1)),
             int(r.integers(c["n_lo"], c["n_hi"] + 1))) for _ in range(c["models"])]


def prepare(case, seed):
    g = _generator(seed)
    s = dict(case=dict(case))
    if case["kind"] == "batched":
        s["problems"] = []
        for W, half, N in _shapes(case):
            H, R = _random_model(W, half, g)
            ef = torch.rand(1, dtype=torch.float64, device="cuda", generator=g) - 0.5
            s["problems"].append((H, R, (N, N, N), ef, 1e-3))
        return s
    H, R = _model(case, g)
    mesh = (case["n1"], case["n2"], case["n3"])
    s.update(H=H, R=R, mesh=mesh, etas=_etas(case))
    if case["kind"] in ("ahc", "ahc_host", "grad"):
        s["E_F"] = _fermi(case, g)
        s["k_range"] = (case["k0"], case["k0"] + case["nk"])
    else:
        s["kidx"] = torch.randint(0, mesh[0] * mesh[1] * mesh[2], (case["nk"],), device="cuda", generator=g)
    if case["kind"] == "ahc_host":
        s["H"], s["E_F"] = H.cpu().numpy(), s["E_F"].cpu().numpy()
    if case["kind"] == "grad":   # the weights of the fitted quantity
        s["g"] = torch.randn((case["n_eta"], case["n_ef"]), dtype=torch.float64, device="cuda", generator=g)
    return s


# --------------------------------------------------------------------------- the calls
def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "ahc":
        return kubo.ahc(s["H"], s["R"], s["mesh"], s["E_F"], etas=s["etas"], kT=c["kT"],
                        precision=c["precision"], k_range=s["k_range"])
    if kind == "ahc_host":
        return kubo.ahc_host(s["H"], s["R"], s["mesh"], s["E_F"], etas=s["etas"], kT=c["kT"],
                             precision=c["precision"], k_range=s["k_range"])
    if kind == "batched":
        return kubo.ahc_batched(s["problems"], precision=c["precision"])[0]
    if kind == "grad":
        H = s["H"].detach().requires_grad_(True)
        S = kubo.AHC.apply(H, s["R"], s["mesh"], s["E_F"], s["etas"][0], s["etas"], c["kT"], s["k_range"])
        (S * s["g"]).sum().backward()
        return S.detach(), H.grad
    if kind == "ahc_k":
        return kubo.ahc_k(s["H"], s["R"], s["mesh"], s["kidx"], etas=s["etas"], precision=c["precision"])
    Hk, X, Y = kubo.bloch(s["H"], s["R"], s["mesh"], s["kidx"], precision=c["precision"])
    E, U = kubo.eigh_batched(Hk, c["W"])
    return Hk, X, Y, E, kubo.berry_batched(E, U, X, Y, etas=s["etas"])


# --------------------------------------------------------------------------- work
def work(case):
    """Inputs read once and outputs written once; operations of the dense Fourier sum over the
    Hermitian half set, the eigensystem and the rotations (the gradient: their adjoint as well)."""
    if case["kind"] == "batched":
        one = [(W, (2 * h + 1) ** 3, N ** 3) for W, h, N in _shapes(case)]
        return dict(bytes=float(sum(16 * n * W * W + 16 for W, n, _ in one)),
                    flops=float(sum(k * _fp64_flops(W, n) for W, n, k in one)))
    W, nk = case["W"], case["nk"]
    N_R = 11 if case["model"] == "haldane" else (2 * case["half"] + 1) ** 3
    flops = nk * _fp64_flops(W, N_R)
    nbytes = 16.0 * N_R * W * W
    if case["kind"] == "grad":
        flops += nk * (6.0 * N_R * W * W + 80.0 * W ** 3)
        nbytes *= 2.0
    if case["kind"] in ("ahc_k", "steps"):
        nbytes += nk * (8.0 + 8.0 * W * (1 + case["n_eta"]))
    if case["kind"] == "steps":
        nbytes += nk * 24.0 * W * W
    if "n_ef" in case:
        nbytes += 8.0 * case["n_ef"] * (1 + case["n_eta"])
    return dict(bytes=nbytes, flops=float(flops))


# --------------------------------------------------------------------------- 64-bit reference
def _bloch64(H, R, mesh, idx):
    """H(k), d_x H(k), d_y H(k) of listed mesh points, phases from exactly reduced angles."""
    N1, N2, N3 = mesh
    j = torch.stack([idx // (N2 * N3), (idx // N3) % N2, idx % N3], 1)
    Rt = torch.from_numpy(np.asarray(R, dtype=np.int64)).cuda()
    turn = torch.zeros((idx.numel(), Rt.shape[0]), dtype=torch.float64, device="cuda")
    for a, n in enumerate(mesh):
        turn += ((j[:, a:a + 1] * Rt[None, :, a]) % n).double() / n
    ph = torch.polar(torch.ones_like(turn), 2.0 * math.pi * turn)
    n, W = Rt.shape[0], H.shape[1]
    flat = H.reshape(n, W * W)
    w = [torch.ones(n, dtype=torch.complex128, device="cuda"), 1j * Rt[:, 0].double(), 1j * Rt[:, 1].double()]
    out = [((ph * x[None, :]) @ flat).reshape(-1, W, W) for x in w]
    return [0.5 * (A + A.conj().transpose(1, 2)) for A in out]


def _curvature64(E, Vx, Vy, etas):
    dE2 = (E[:, :, None] - E[:, None, :]) ** 2
    num = -2.0 * (Vx * Vy.transpose(1, 2)).imag
    off = 1.0 - torch.eye(E.shape[1], dtype=torch.float64, device="cuda")
    return torch.stack([(num * off / (dE2 + eta * eta + (1.0 - off))).sum(2) for eta in etas])


def _bands64(H, R, mesh, idx, etas):
    Hk, X, Y = _bloch64(H, R, mesh, idx)
    E, U = torch.linalg.eigh(Hk)
    Uh = U.conj().transpose(1, 2)
    return E, _curvature64(E, Uh @ X @ U, Uh @ Y @ U, etas), (Hk, X, Y)


def _occupation64(E, ef, kT):
    if kT == 0.0:
        return (E[None] < ef[:, None, None]).double()
    return torch.sigmoid((ef[:, None, None] - E[None]) / kT)


def _sum64(H, R, mesh, k0, nk, ef, etas, kT, g=None):
    """S, and with weights g the gradient of sum(g S) with respect to H(R)."""
    W, n = H.shape[1], len(R)
    S = torch.zeros((len(etas), ef.numel()), dtype=torch.float64, device="cuda")
    step = max(1, min(4096 if W > 8 else 32768, int(2e8 / (n + W * W * 6 + W * ef.numel()))))
    H = H.detach().requires_grad_(g is not None)
    for a in range(k0, k0 + nk, step):
        idx = torch.arange(a, min(a + step, k0 + nk), device="cuda")
        E, Om, _ = _bands64(H, R, mesh, idx, etas)
        one = torch.einsum("jkn,ekn->ej", _occupation64(E, ef, kT), Om) / float(mesh[0] * mesh[1] * mesh[2])
        if g is not None:
            (one * g).sum().backward()
        S += one.detach()
    return S if g is None else (S, H.grad)


def _packed(A):
    """Real parts of the upper triangle, imaginary parts of the strict one mirrored below."""
    up = torch.triu(torch.ones(A.shape[1:], dtype=torch.bool, device="cuda"))
    return torch.where(up, A.real, A.imag.transpose(1, 2)).reshape(A.shape[0], -1)


def _eigh_seconds(W, count):
    """What torch's batched eigensystems take (one matrix at a time above order 32)."""
    return count * (6e-5 * W if W > 32 else 2e-4 if W > 8 else 8e-5)


def exact(case, seed):
    kind = case["kind"]
    sizes = [(W, N ** 3) for W, _, N in _shapes(case)] if kind == "batched" else [(case["W"], case["nk"])]
    if sum(_eigh_seconds(W, n) * (2.0 if kind == "grad" else 1.0) for W, n in sizes) > 16.0:
        return None
    s = prepare(case, seed)
    if kind in ("ahc", "ahc_host"):
        H, ef = (torch.as_tensor(s[k], device="cuda") for k in ("H", "E_F"))
        S = _sum64(H, s["R"], s["mesh"], case["k0"], case["nk"], ef, s["etas"], case["kT"])
        return S.cpu().numpy() if kind == "ahc_host" else S
    if kind == "grad":
        return _sum64(s["H"], s["R"], s["mesh"], case["k0"], case["nk"], s["E_F"], s["etas"], case["kT"], s["g"])
    if kind == "batched":
        return [_sum64(H, R, mesh, 0, mesh[0] * mesh[1] * mesh[2], ef, [eta], 0.0)
                for H, R, mesh, ef, eta in s["problems"]]
    parts = [_bands64(s["H"], s["R"], s["mesh"], i, s["etas"]) for i in s["kidx"].split(512)]
    E, Om = torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts], 1)
    if kind == "ahc_k":
        return E, Om
    Hk, X, Y = (_packed(torch.cat([p[2][q] for p in parts])) for q in range(3))
    return Hk, X, Y, E, Om
