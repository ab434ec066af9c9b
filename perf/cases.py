"""The calls that the framework's speed is measured on.

A case is one pass through a public entry point of the package, as a program
that holds the plan, the orbitals and the output buffers makes it: an electronic
structure code builds the ACE operator once per outer iteration, applies it to
blocks of bands many times, solves Poisson problems for the density, and asks
for the exchange energy and its gradient. Sizes follow the workloads of
`synth.py`, the tests and the benchmark: a grid spacing of 20.5/48 bohr, grids
from 16^3 to 96^3, 1 to 1024 exchange orbitals, 1 to 1536 bands.

Orbitals are seeded band-limited fields (plane waves of a 10 Ha sphere with
Gaussian-decaying random coefficients), orthonormalised on the grid; targets
are the same fields, normalised.
"""
import math

import torch

H = 20.5 / 48            # grid spacing of every workload (bohr)
ECUT = 10.0              # plane-wave sphere of the orbitals (Ha)
OMEGA = 0.106            # screening parameter of the erfc workloads
CDTYPE = {"c64": torch.complex64, "c128": torch.complex128, "r64": torch.float64}
EDGES = (16, 20, 24, 32, 36, 40, 48, 64, 96)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one Hartree potential of one density, once per density update: the smallest call
        dict(name="poisson_48_b1", kind="poisson", grid="48", nb=1, dtype="c64", kernel="bare"),
        # a small molecule at the Gamma point in FP64: real orbitals, launch-bound
        dict(name="build_r64_24_n8", kind="build", grid="24", n_occ=8, dtype="r64", kernel="bare"),
        # one application of the model Hamiltonian (kinetic, local, V_ACE) to a subspace block:
        # the call an eigensolver makes hundreds of times, eager launches on fresh tensors
        dict(name="hamiltonian_48_n16_b24", kind="hamiltonian", grid="48", n_occ=16, nb=24, dtype="c64"),
        # the ACE apply on every band of a 64-atom cell
        dict(name="apply_48_n128_b192", kind="apply", grid="48", n_occ=128, nb=192, dtype="c64"),
        # the exact exchange operator on a block of unoccupied bands, orthorhombic cell, odd counts
        dict(name="vx_48x40x36_n61_b37", kind="vx", grid="48x40x36", n_occ=61, nb=37, dtype="c64", kernel="erfc"),
        # the ACE construction of a 64-atom cell, screened kernel
        dict(name="build_48_n128", kind="build", grid="48", n_occ=128, dtype="c64", kernel="erfc"),
        # the same construction in FP64 (the precision of the model SCF's default), odd count
        dict(name="build_c128_32_n27", kind="build", grid="32", n_occ=27, dtype="c128", kernel="bare"),
        # oversampled construction: the operator exact on unoccupied orbitals too
        dict(name="oversampled_40_n45_p70", kind="oversampled", grid="40", n_occ=45, n_phi=70, dtype="c64",
             kernel="erfc"),
        # uneven systems built as one batch
        dict(name="batch_8_uneven", kind="batch", systems="36:55,32:102,36:40,64:34,48:121,32:39,40:35,24:17"),
        # exchange energy and its gradient (forward and backward of the autograd function)
        dict(name="energy_grad_64_n96", kind="energy_grad", grid="64", n_occ=96, dtype="c64", kernel="bare"),
        # construction on the largest grid
        dict(name="build_96_n128", kind="build", grid="96", n_occ=128, dtype="c64", kernel="erfc"),
        # the ACE apply on every band of a 512-atom cell: the largest apply
        dict(name="apply_96_n1024_b1536", kind="apply", grid="96", n_occ=1024, nb=1536, dtype="c64"),
    ]


def _log(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# orthorhombic grids: compiled planes and square planes with another pencil length
_ORTHO = ("12x16x20", "16x24x12", "24x16x36", "40x48x36", "48x40x64", "16x16x64", "32x32x48", "48x48x96", "64x64x40")


def _grid_cost(g):
    nx, ny, nz = _dims(g)
    return nx * ny * nz


def draw(rng):
    kind = rng.choice(["poisson", "build", "build", "build64", "hamiltonian", "apply", "apply", "vx", "oversampled",
                       "batch", "energy_grad"])
    grid = rng.choice(_ORTHO) if rng.random() < 0.25 else str(rng.choice(EDGES))
    kernel = rng.choice(["bare", "erfc"])
    ng = _grid_cost(grid)
    if kind == "poisson":
        dtype = rng.choice(["c64", "c64", "c128", "r64"])
        return dict(kind=kind, grid=grid, nb=_log(rng, 1, min(192, 60_000_000 // ng)), dtype=dtype, kernel=kernel)
    if kind == "build64":     # FP64 plans: small grids and counts
        grid = str(rng.choice((12, 16, 20, 24, 32)))
        return dict(kind="build", grid=grid, n_occ=_log(rng, 2, 32), dtype=rng.choice(["c128", "r64"]), kernel=kernel)
    if kind == "hamiltonian":
        edge = rng.choice((16, 20, 24, 32, 36, 40, 48))
        n = _log(rng, 4, 64)
        return dict(kind=kind, grid=str(edge), n_occ=n, nb=n + max(2, n // 2), dtype=rng.choice(["c64", "c64", "c128"]))
    if kind == "apply":
        n = _log(rng, 8, min(1024, 500_000_000 // ng))
        nb = _log(rng, 1, min(1536, 700_000_000 // ng))
        return dict(kind=kind, grid=grid, n_occ=n, nb=nb, dtype="c64")
    most = min(256, int(math.sqrt(2 * 4.0e9 / ng)))   # pair solves x points within the largest construction
    if kind == "vx":
        n = _log(rng, 4, most)
        return dict(kind=kind, grid=grid, n_occ=n, nb=_log(rng, 1, max(1, most // 2)), dtype="c64", kernel=kernel)
    if kind == "oversampled":
        n = _log(rng, 4, max(8, most // 2))
        return dict(kind=kind, grid=grid, n_occ=n, n_phi=n + _log(rng, 1, max(2, n // 2)), dtype="c64", kernel=kernel)
    if kind == "batch":
        count = rng.randint(2, 8)
        return dict(kind=kind, systems=",".join(f"{rng.choice((24, 32, 36, 40, 48, 64))}:{rng.randint(8, 96)}"
                                                for _ in range(count)))
    if kind == "energy_grad":
        most = min(most, int(math.sqrt(2 * 1.2e9 / ng)))   # the pair potentials of three states fit the card
        return dict(kind=kind, grid=grid, n_occ=_log(rng, 4, most), dtype="c64", kernel=kernel)
    return dict(kind="build", grid=grid, n_occ=_log(rng, 4, most), dtype="c64", kernel=kernel)


# ------------------------------------------------------------------ geometry
def _dims(grid):
    """'48' or 'n_x x n_y x n_z' -> (n_x, n_y, n_z)."""
    v = [int(t) for t in str(grid).split("x")]
    return (v[0],) * 3 if len(v) == 1 else tuple(v)


def _cell(dims):
    return tuple(H * n for n in dims)


def _dv(dims):
    return H ** 3


def _g2(dims, dtype=torch.float64):
    nx, ny, nz = dims
    ax = [2 * math.pi * torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64) / l
          for n, l in zip(dims, _cell(dims))]
    return (ax[2][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[0][None, None, :] ** 2).to(dtype)


# ------------------------------------------------------------------ inputs
def _fields(dims, count, seed, dtype):
    """`count` band-limited random fields (count, n_z, n_y, n_x), normalised."""
    nx, ny, nz = dims
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rt = torch.float32 if dtype == "c64" else torch.float64
    g2 = _g2(dims)
    decay = torch.where(0.5 * g2 <= ECUT, torch.exp(-g2 / (2 * ECUT)), torch.zeros_like(g2)).to(rt)
    out = torch.empty((count, nz, ny, nx), dtype=CDTYPE[dtype], device="cuda")
    step = max(1, min(count, 60_000_000 // (nx * ny * nz)))
    for i in range(0, count, step):
        k = min(step, count - i)
        c = torch.randn((k, nz, ny, nx, 2), generator=gen, device="cuda", dtype=rt)
        f = torch.fft.ifftn(torch.view_as_complex(c) * decay, dim=(1, 2, 3))
        f = f.real.contiguous() if dtype == "r64" else f
        nrm = torch.linalg.vector_norm(f.reshape(k, -1), dim=1) * math.sqrt(_dv(dims))
        out[i:i + k] = f / nrm[:, None, None, None]
    return out


def _orthonormal(x, dims):
    """Orthonormal in dV sum conj(f) g: x <- L^{-1} x with x x^* = L L^* (rows are vectors)."""
    m = x.reshape(x.shape[0], -1)
    wide = torch.complex128 if x.is_complex() else torch.float64
    for _ in range(2):
        g = (m.conj() @ m.T).to(wide).conj() * _dv(dims)
        l = torch.linalg.cholesky(g)
        m = torch.linalg.solve_triangular(l, torch.eye(l.shape[0], dtype=wide, device="cuda"), upper=False).to(x.dtype) @ m
    return m.reshape(x.shape).contiguous()


def _orbitals(dims, count, seed, dtype):
    return _orthonormal(_fields(dims, count, seed, dtype), dims)


def _operator(dims, count, seed, dtype):
    """Vectors with the size of the ACE operator's: V_ACE = -sum |xi><xi| with exchange
    eigenvalues of 0.05 to 0.8 Ha."""
    x = _fields(dims, count, seed, dtype)
    gen = torch.Generator(device="cuda").manual_seed(seed + 7)
    s = torch.sqrt(0.05 + 0.75 * torch.rand(count, generator=gen, device="cuda", dtype=torch.float64))
    x *= s[:, None, None, None].to(x.real.dtype)
    return x


def _systems(text):
    return [(int(a), int(b)) for a, b in (t.split(":") for t in text.split(","))]


def _well(dims):
    """A smooth attractive local potential (Hartree) on the grid."""
    ax = [torch.cos(2 * math.pi * torch.arange(n, device="cuda", dtype=torch.float64) / n) for n in dims]
    return -0.4 * (ax[2][:, None, None] + ax[1][None, :, None] + ax[0][None, None, :])


def _plan(case, n_occ, kernel=None):
    from paper_1601_07159_gb300 import ace
    dims = _dims(case["grid"])
    kernel = kernel or case["kernel"]
    return ace.Plan(dims, _cell(dims), n_occ, dtype=case["dtype"], kernel=kernel,
                    omega=OMEGA if kernel == "erfc" else 0.0)


def _inputs(case, seed):
    """The arrays of a case, from the seed alone."""
    kind = case["kind"]
    seed = 1601071590 + 1013 * int(seed)
    if kind == "batch":
        return {"phis": [_orbitals((n,) * 3, N, seed + i, "c64") for i, (n, N) in enumerate(_systems(case["systems"]))]}
    dims, dtype = _dims(case["grid"]), case["dtype"]
    if kind == "poisson":     # densities: sums of squares of orbitals
        f = _fields(dims, case["nb"], seed, dtype)
        return {"rho": (f.abs() ** 2).to(CDTYPE[dtype])}
    if kind == "hamiltonian":
        return {"xi": _operator(dims, case["n_occ"], seed, dtype), "psi": _orbitals(dims, case["nb"], seed + 500, dtype),
                "v": _well(dims)}
    if kind == "apply":
        return {"xi": _operator(dims, case["n_occ"], seed, dtype), "psi": _fields(dims, case["nb"], seed + 500, dtype)}
    if kind == "vx":
        return {"phi": _orbitals(dims, case["n_occ"], seed, dtype), "psi": _fields(dims, case["nb"], seed + 500, dtype)}
    return {"phi": _orbitals(dims, case["n_phi"] if kind == "oversampled" else case["n_occ"], seed, dtype)}


def prepare(case, seed):
    """Plan, inputs and output buffers: what a program keeps between calls."""
    from paper_1601_07159_gb300 import ace, scf
    st = dict(case=case, **_inputs(case, seed))
    kind = case["kind"]
    if kind == "batch":
        st["batch"] = ace.Batch([ace.Plan(n, H * n, N, dtype="c64", kernel="bare") for n, N in _systems(case["systems"])])
        st["xis"] = [torch.empty_like(p) for p in st["phis"]]
    elif kind == "hamiltonian":
        dims = _dims(case["grid"])
        st["model"] = scf.ModelHF(dims[0], H * dims[0], case["n_occ"], st["v"], dtype=case["dtype"])
        st["v_eff"] = st["model"].v_loc
    elif kind == "poisson":
        st["plan"] = _plan(case, 1)
        st["out"] = torch.empty_like(st["rho"])
    elif kind == "apply":
        st["plan"] = _plan(case, case["n_occ"], "bare")
        st["out"] = torch.empty_like(st["psi"])
    elif kind == "vx":
        st["plan"] = _plan(case, case["n_occ"])
        st["out"] = torch.empty_like(st["psi"])
    else:
        st["plan"] = _plan(case, case["n_occ"])
        if kind == "energy_grad":
            st["phi"].requires_grad_(True)
        else:
            st["xi"], st["w"] = torch.empty_like(st["phi"]), torch.empty_like(st["phi"])
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    kind = st["case"]["kind"]
    if kind == "poisson":
        return st["plan"].poisson(st["rho"], out=st["out"])
    if kind == "build":
        return st["plan"].build(st["phi"], xi=st["xi"], w=st["w"])
    if kind == "oversampled":
        return st["plan"].build_oversampled(st["phi"], xi=st["xi"], w=st["w"])
    if kind == "apply":
        return st["plan"].apply(st["xi"], st["psi"], out=st["out"])
    if kind == "vx":
        return st["plan"].exchange_apply(st["phi"], st["psi"], out=st["out"])
    if kind == "hamiltonian":
        return st["model"].apply(st["psi"], st["v_eff"], xi=st["xi"])
    if kind == "batch":
        xis, ex = st["batch"].build(st["phis"], st["xis"])
        return {"Xi": xis, "Ex": ex}
    from paper_1601_07159_gb300 import ace
    ex = ace.exchange_energy(st["phi"], st["plan"])
    (grad,) = torch.autograd.grad(ex, st["phi"])
    return {"Ex": ex.detach(), "grad": grad}


# ------------------------------------------------------------------ the work a pass cannot do without
def _solve_flops(ng, real=False):
    """One pair: product, forward and inverse transform, kernel, both accumulations."""
    fft = 5.0 * ng * math.log2(ng)
    return (1.0 if real else 2.0) * fft + (8.0 if real else 24.0) * ng


def _build_work(ng, n_occ, n_phi, esize, real):
    pairs = n_occ * (n_occ + 1) / 2 + n_occ * (n_phi - n_occ)
    mac = 2.0 if real else 8.0
    # Phi read once, W and Xi written; M and Xi = W L^{-*} (triangular) in the vectors' arithmetic
    flops = pairs * _solve_flops(ng, real) + 1.5 * mac * n_phi * n_phi * ng + 0.5 * mac * n_phi ** 3
    return 3.0 * n_phi * ng * esize, flops


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for n, N in _systems(case["systems"]):
            bb, ff = _build_work(n ** 3, N, N, 8, False)
            b += bb * 2 / 3          # Phi in, Xi out
            f += ff
        return {"bytes": b, "flops": f}
    nx, ny, nz = _dims(case["grid"])
    ng = nx * ny * nz
    real = case["dtype"] == "r64"
    es = 8 if case["dtype"] in ("c64", "r64") else 16
    if kind == "poisson":
        nb = case["nb"]
        return {"bytes": 2.0 * nb * ng * es, "flops": nb * ((1 if real else 2) * 5.0 * ng * math.log2(ng) + 2.0 * ng)}
    if kind in ("apply", "hamiltonian"):
        N, nb = case["n_occ"], case["nb"]
        b, f = (N + 2.0 * nb) * ng * es, 16.0 * N * nb * ng
        if kind == "hamiltonian":
            f += nb * (10.0 * ng * math.log2(ng) + 8.0 * ng)
        return {"bytes": b, "flops": f}
    if kind == "vx":
        N, nb = case["n_occ"], case["nb"]
        return {"bytes": (N + 2.0 * nb) * ng * es, "flops": N * nb * _solve_flops(ng)}
    if kind == "energy_grad":
        N = case["n_occ"]
        return {"bytes": 2.0 * N * ng * es, "flops": N * (N + 1) / 2 * (_solve_flops(ng) + 4.0 * ng)}
    b, f = _build_work(ng, case["n_occ"], case.get("n_phi", case["n_occ"]), es, real)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in 64 bits, plain torch
def _kernel64(dims, kernel):
    g2 = _g2(dims)
    zero = g2 == 0
    safe = torch.where(zero, torch.ones_like(g2), g2)
    if kernel == "kinetic":
        return 0.5 * g2
    k = 4 * math.pi / safe
    if kernel == "erfc":
        k = k * -torch.expm1(-safe / (4 * OMEGA ** 2))
        return torch.where(zero, torch.full_like(k, math.pi / OMEGA ** 2), k)
    return torch.where(zero, torch.zeros_like(k), k)


def _solve64(rho, k):
    return torch.fft.ifftn(torch.fft.fftn(rho, dim=(1, 2, 3)).mul_(k), dim=(1, 2, 3))


def _vx64(phi, psi, k):
    """(V_X[phi] psi)_b = -sum_j phi_j Poisson[conj(phi_j) psi_b]."""
    out = torch.zeros_like(psi)
    step = max(1, 30_000_000 // phi[0].numel())
    for b in range(psi.shape[0]):
        for j in range(0, phi.shape[0], step):
            p = phi[j:j + step]
            out[b] -= (p * _solve64(p.conj() * psi[b], k)).sum(0)
    return out


def _vx_sym64(phi, k):
    """V_X[phi] phi over the unique pairs (v_ij = conj(v_ji))."""
    out = torch.zeros_like(phi)
    step = max(1, 30_000_000 // phi[0].numel())
    for i in range(phi.shape[0]):
        for j in range(i, phi.shape[0], step):
            q = phi[j:j + step]
            v = _solve64(phi[i].conj() * q, k)             # conj(phi_i) phi_j
            out[j:j + step] -= phi[i] * v
            lo = 1 if j == i else 0
            out[i] -= (q[lo:] * v[lo:].conj()).sum(0)
    return out


def _ace64(phi, w, dims):
    p, m = phi.reshape(phi.shape[0], -1), w.reshape(w.shape[0], -1)
    M = _dv(dims) * (p.conj() @ m.T)
    M = 0.5 * (M + M.conj().T)
    l = torch.linalg.cholesky(-M)
    # Xi = W L^{-*}; the vectors are rows here, so Xi^T = (L^{-*})^T W^T = conj(L)^{-1} W^T
    xi = torch.linalg.solve_triangular(l.conj(), m, upper=False)
    return M, xi.reshape(w.shape)


def _apply64(xi, psi, dims):
    x, p = xi.reshape(xi.shape[0], -1), psi.reshape(psi.shape[0], -1)
    c = _dv(dims) * (x.conj() @ p.T)                       # N x nb
    return -(c.T @ x).reshape(psi.shape)


def exact(case, seed):
    kind = case["kind"]
    w = work(case)["flops"]
    if kind == "apply" and w > 6e12:                       # over 20 s in 64 bits
        return None
    inp = _inputs(case, seed)
    if kind == "batch":
        xis, ex = [], []
        for (n, N), phi in zip(_systems(case["systems"]), inp["phis"]):
            phi = phi.to(torch.complex128)
            W = _vx_sym64(phi, _kernel64((n,) * 3, "bare"))
            M, xi = _ace64(phi, W, (n,) * 3)
            xis.append(xi)
            ex.append(0.5 * torch.diagonal(M).real.sum())
        return {"Xi": xis, "Ex": torch.stack(ex)}
    dims = _dims(case["grid"])
    wide = torch.float64 if case["dtype"] == "r64" else torch.complex128
    if kind == "poisson":
        v = _solve64(inp["rho"].to(torch.complex128), _kernel64(dims, case["kernel"]))
        return v.real.contiguous() if case["dtype"] == "r64" else v
    if kind == "apply":
        return _apply64(inp["xi"].to(wide), inp["psi"].to(wide), dims)
    if kind == "hamiltonian":
        psi = inp["psi"].to(wide)
        v = inp["v"].to(torch.float32 if case["dtype"] == "c64" else torch.float64).to(torch.float64)
        return _solve64(psi, _kernel64(dims, "kinetic")) + v * psi + _apply64(inp["xi"].to(wide), psi, dims)
    k = _kernel64(dims, case["kernel"])
    if kind == "vx":
        return _vx64(inp["phi"].to(wide), inp["psi"].to(wide), k)
    phi = inp["phi"].detach().to(torch.complex128)
    real = case["dtype"] == "r64"
    if kind == "energy_grad":
        W = _vx_sym64(phi, k)
        e = 0.5 * _dv(dims) * (phi.conj() * W).real.sum()
        return {"Ex": e, "grad": 2 * _dv(dims) * W}
    n_occ = case["n_occ"]
    W = _vx_sym64(phi[:n_occ], k)
    if kind == "oversampled":
        W = torch.cat([W, _vx64(phi[:n_occ], phi[n_occ:], k)])
    if real:
        phi, W = phi.real.contiguous(), W.real.contiguous()
    M, xi = _ace64(phi, W, dims)
    return {"Xi": xi, "W": W, "M": M, "Ex": 0.5 * torch.diagonal(M).real[:n_occ].sum()}
