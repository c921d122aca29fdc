"""Timed cases of the library's public entry points, over the sizes it is used at.

Every case is one call (or the two calls that belong together) a user's program makes through
paper_1005_0088_gb300: a density sweep on either precision path, a share of one divided among
ranks, Green functions at chosen points, the energy density matrix, the density of states, a
batched sweep over uneven systems, a chemical-potential search, solves with the factors, and the
training of the chemical-potential network.

Inputs follow the synthetic lattice recipe of the repository: atoms on an integer grid (atom =
x + nx (y + ny z)), 1D nearest neighbours, 2D nearest and next-nearest, 3D all 26 neighbours;
onsite block diag(U(-1, 1)) + symmetrised N(0, 0.1^2), neighbour blocks N(0, 0.1^2), overlap I + c U(-1, 1) on
neighbour blocks with c = min(0.05, 0.75 / largest row sum).  They are drawn on the GPU from the seed.
"""
import functools
import itertools
import math

import numpy as np
import torch

import paper_1005_0088_gb300 as nd

DEV = "cuda"
MU = -0.12                 # chemical potential of the benchmark's sweeps (Ha)
WORKSPACE = 64 << 30       # workspace a program with several plans on one card gives each of them
EXACT_MAX_N = 6600         # largest system whose dense 64-bit route takes a few seconds


def listed():
    return [
        # The smallest sweep: the 1D chain of 64 atoms x 8 orbitals, 40 poles.  Few, tiny fronts: latency and launches count.
        dict(name="chain_fp64", kind="density", nx=64, ny=1, nz=1, orb=8, split=False, poles=40, kT=0.01),
        # The 2D sheet of 32 x 32 atoms on the plain FP64 path.
        dict(name="sheet_fp64", kind="density", nx=32, ny=32, nz=1, orb=4, split=False, poles=80, kT=0.01),
        # The same sheet in split precision, tuned once, as a program that sweeps a geometry many times has it.
        dict(name="sheet_split", kind="density", nx=32, ny=32, nz=1, orb=4, split=True, tune=True, poles=80, kT=0.01),
        # Green functions of a ragged 3D box at eight contour points: factor and selected inversion in FP64, G returned.
        dict(name="box_green", kind="green", nx=9, ny=8, nz=7, orb=5, split=False, points=8),
        # Density and energy density matrix (forces) of a 3D box in split precision.
        dict(name="box_energy", kind="energy", nx=12, ny=11, nz=9, orb=4, split=True, poles=80, kT=0.01),
        # Density of states of a ragged sheet with five orbitals per atom on an energy grid.
        dict(name="sheet_dos", kind="dos", nx=30, ny=26, nz=1, orb=5, split=True, points=81, eta=0.02),
        # The 3D cubic lattice of 16^3 atoms x 4 orbitals, 80 poles, split precision: wide separators.
        dict(name="cubic_split", kind="density", nx=16, ny=16, nz=16, orb=4, split=True, poles=80, kT=0.01),
        # One rank's quarter of a 160-pole sweep of a 3D metallic lattice (8 orbitals, kT 0.002), the widest fronts.
        dict(name="metallic_share", kind="share", nx=16, ny=16, nz=16, orb=8, split=True, poles=160, kT=0.002, rank=0, world=4),
        # Four systems of uneven size in one batched plan, 120 poles, split precision.
        dict(name="batch_split", kind="batched", split=True, poles=120, kT=0.01,
             systems="512x1x1x4 32x32x1x4 30x27x1x5 8x8x8x4"),
        # A whole chemical-potential search on a small sheet: the density of states, then one sweep per trial.
        dict(name="sheet_mu", kind="mu", nx=16, ny=15, nz=1, orb=3, split=False, poles=60, kT=0.01),
        # Sixteen right-hand sides solved with the factors of one shift (a step of the eigensolver's iteration).
        dict(name="box_solve", kind="solve", nx=12, ny=12, nz=11, orb=4, split=False, rhs=16),
        # Training the chemical-potential network on 2000 systems' features (25 of its full-batch steps).
        dict(name="mlp_train", kind="mlp", samples=2000, steps=25),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice(rng, dims, lo, hi):
    if dims == 1:
        return dict(nx=_log_int(rng, lo, hi), ny=1, nz=1)
    if dims == 2:
        return dict(nx=rng.randint(lo, hi), ny=rng.randint(lo, hi), nz=1)
    return dict(nx=rng.randint(lo, hi), ny=rng.randint(lo, hi), nz=rng.randint(lo, hi))


def draw(rng):
    """One more case of the same kinds; flop limits keep it below the largest listed one."""
    while True:
        kind = rng.choice(["density", "density", "density", "green", "energy", "dos", "share", "batched", "mu", "solve", "mlp"])
        if kind == "mlp":
            return dict(kind=kind, samples=_log_int(rng, 64, 4000), steps=rng.randint(5, 40))
        split = rng.random() < 0.6
        if kind == "batched":
            parts = []
            for _ in range(rng.randint(2, 5)):
                dims = rng.randint(1, 3)
                g = _lattice(rng, dims, *((32, 512), (8, 32), (4, 8))[dims - 1])
                parts.append("%dx%dx%dx%d" % (g["nx"], g["ny"], g["nz"], rng.randint(3, 6)))
            case = dict(kind=kind, split=True, poles=rng.randint(40, 120), kT=0.01, systems=" ".join(parts))
        else:
            dims = 3 if kind == "share" else rng.randint(1, 3)
            hi3 = 16 if split and kind != "green" else 9      # a green case holds the factors of all its points
            case = dict(kind=kind, **_lattice(rng, dims, *((16, 1024), (8, 48 if split else 32), (4, hi3))[dims - 1]))
            case.update(orb=rng.randint(3, 8), split=split)
            if kind in ("density", "energy", "mu", "share"):
                case.update(poles=rng.randint(40, 80), kT=0.01)
            if kind == "density" and split and dims == 2:
                case.update(tune=True)
            if kind == "share":
                case.update(split=True, poles=160, kT=0.002, world=rng.randint(3, 8))
                case.update(rank=rng.randrange(case["world"]))
            if kind == "mu":
                case.update(split=False)
            if kind in ("green", "dos"):
                case.update(points=rng.randint(4, 16) if kind == "green" else rng.randint(20, 81))
            if kind == "dos":
                case.update(eta=0.02)
            if kind == "solve":
                case.update(split=False, rhs=rng.randint(1, 32))
        limit = 1.5e13 if case["split"] else 1.5e11
        if kind in ("mu", "solve"):
            limit = 5e11
        if work(case)["flops"] <= limit:
            return case


# ------------------------------------------------------------------------------------ inputs ---
class Lattice:
    """Pattern and geometry of a lattice, and where each block's elements stand in the CSR arrays."""

    def __init__(self, nx, ny, nz, orb):
        dims = 3 if nz > 1 else 2 if ny > 1 else 1
        if dims == 1:
            offs = [(1, 0, 0)]
        elif dims == 2:
            offs = [(1, 0, 0), (0, 1, 0), (1, 1, 0), (1, -1, 0)]
        else:
            offs = [d for d in itertools.product((-1, 0, 1), repeat=3) if d > (0, 0, 0)]
        na, o = nx * ny * nz, orb
        z, y, x = (v.ravel() for v in np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij"))
        pa, pb = [], []
        for dx, dy, dz in offs:
            x2, y2, z2 = x + dx, y + dy, z + dz
            ok = (x2 >= 0) & (x2 < nx) & (y2 >= 0) & (y2 < ny) & (z2 >= 0) & (z2 < nz)
            pa.append(np.flatnonzero(ok))
            pb.append((x2 + nx * (y2 + ny * z2))[ok])
        pa, pb = np.concatenate(pa), np.concatenate(pb)
        # blocks sorted by (row atom, column atom)
        ba = np.concatenate([np.arange(na), pa, pb])
        bb = np.concatenate([np.arange(na), pb, pa])
        order = np.argsort(ba * na + bb, kind="stable")
        place = np.empty_like(order)
        place[order] = np.arange(order.size)
        deg = np.bincount(ba, minlength=na)
        first = np.concatenate([[0], np.cumsum(deg)])
        start = o * o * first[ba] + (place - first[ba]) * o      # element (0, 0) of each block
        step = deg[ba] * o                                       # from one row of the block to the next
        self.n, self.nnz, self.orb, self.n_pairs = na * o, int(first[-1]) * o * o, o, pa.size
        self.rowptr = np.concatenate([[0], np.cumsum(np.repeat(deg * o, o))]).astype(np.int64)
        col = (bb[order][:, None] * o + np.arange(o)).reshape(-1)
        cut = np.repeat(first[:-1] * o, o), np.repeat(first[1:] * o, o)
        idx = np.arange(self.nnz) - np.repeat(self.rowptr[:-1] - cut[0], np.diff(self.rowptr))
        self.col = col[idx].astype(np.int32)
        self.centers = np.stack([x, y, z], axis=1).astype(np.float64)
        self.atom_of_basis = np.repeat(np.arange(na, dtype=np.int32), o)
        self.na, self.pa, self.pb = na, pa, pb
        k = np.arange(o)
        pos = start[:, None, None] + step[:, None, None] * k[None, :, None] + k[None, None, :]
        self.pos = pos

    def values(self, gen):
        """H and S on the pattern, on the GPU."""
        o, na, npair = self.orb, self.na, self.n_pairs
        pos = torch.as_tensor(self.pos, device=DEV)

        def uniform(*shape):
            return 2.0 * torch.rand(*shape, generator=gen, device=DEV, dtype=torch.float64) - 1.0

        g = 0.1 * torch.randn(na, o, o, generator=gen, device=DEV, dtype=torch.float64)
        on = 0.5 * (g + g.transpose(1, 2)) + torch.diag_embed(uniform(na, o))
        hop = 0.1 * torch.randn(npair, o, o, generator=gen, device=DEV, dtype=torch.float64)
        w = uniform(npair, o, o)
        # row sums on the host: a fixed order of additions, so that a seed gives the same values to the last bit
        k = np.arange(o)
        at = np.concatenate([(self.pa[:, None] * o + k).ravel(), (self.pb[:, None] * o + k).ravel()])
        sums = torch.cat([w.abs().sum(2), w.abs().sum(1)]).reshape(-1).cpu().numpy()
        top = float(np.bincount(at, weights=sums, minlength=1).max())
        w = w * min(0.05, 0.75 / max(top, 1e-300))
        H = torch.empty(self.nnz, device=DEV, dtype=torch.float64)
        S = torch.empty_like(H)
        eye = torch.eye(o, device=DEV, dtype=torch.float64).expand(na, o, o)
        for out, a, b in ((H, on, hop), (S, eye, w)):
            out[pos.reshape(-1)] = torch.cat([a, b, b.transpose(1, 2)]).reshape(-1)
        return H, S


@functools.lru_cache(maxsize=8)
def _geometry(nx, ny, nz, orb):
    return Lattice(nx, ny, nz, orb)


def _parts(case):
    """The lattices of a case (one, but for a batched plan)."""
    if case["kind"] == "batched":
        return [_geometry(*(int(v) for v in s.split("x"))) for s in case["systems"].split()]
    return [_geometry(case["nx"], case["ny"], case["nz"], case["orb"])]


def _options(case):
    return dict(precision=nd.NDSI_PREC_SPLIT if case["split"] else nd.NDSI_PREC_FP64, max_workspace_bytes=WORKSPACE)


def _plan(case):
    parts = _parts(case)
    if case["kind"] == "batched":
        return nd.analyze_batched(parts, **_options(case))
    return nd.analyze_system(parts[0], **_options(case))


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1005008800 + int(seed))
    return g


def _points(case):
    """Green-function points: the lowest Matsubara-like points above MU, or the eigensolver's kind of shift."""
    if case["kind"] == "solve":
        return np.array([MU + 0.01j])
    return MU + 1j * math.pi * 0.01 * (2 * np.arange(case["points"]) + 1)


def _energies(case):
    return np.linspace(-1.5, 1.5, case["points"])


def _mlp_inputs(case, seed):
    """Features and targets of the network's kind: 24 + 6 Chebyshev moments in [-1, 1] that fall off with the order, a filling and 10 kT."""
    gen = _generator(seed)
    n = case["samples"]
    fall = torch.cat([0.5 ** (0.25 * torch.arange(24)), 0.4 ** torch.arange(1, 7).double()]).to(DEV).double()
    x = torch.empty(n, 32, device=DEV, dtype=torch.float64)
    x[:, :30] = fall * torch.randn(n, 30, generator=gen, device=DEV, dtype=torch.float64).clamp(-2, 2) * 0.5
    x[:, 30] = 0.15 + 0.7 * torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    x[:, 31] = 0.05 + 0.15 * torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
    t = 1.6 * (x[:, 30] - 0.5) + x[:, 0] - 0.3 * x[:, 1] * x[:, 30] + 0.02 * torch.randn(n, generator=gen, device=DEV, dtype=torch.float64)
    params = torch.zeros(nd.NDSI_MLP_PARAMS, device=DEV, dtype=torch.float32)
    nd.ndsi_mlp_init(params, 7 + int(seed))
    return params, x.float().contiguous(), t.float().contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        params, x, t = _mlp_inputs(case, seed)
        return dict(case=case, start=params, params=params.clone(), X=x, T=t)
    gen = _generator(seed)
    parts = _parts(case)
    hs = [p.values(gen) for p in parts]
    H = torch.cat([h for h, _ in hs]) if len(hs) > 1 else hs[0][0]
    S = torch.cat([s for _, s in hs]) if len(hs) > 1 else hs[0][1]
    state = dict(case=case, plan=_plan(case), H=H, S=S)
    if kind in ("density", "share", "energy", "mu", "batched"):
        state["rho"] = torch.zeros_like(H)
        state["ne"] = torch.zeros(len(parts), device=DEV, dtype=torch.float64)
    if kind == "energy":
        state["e"] = torch.zeros_like(H)
    if kind == "share":
        state["share"] = nd.ndsi_pole_shard(case["poles"], case["rank"], case["world"])
    if kind == "green":
        state["G"] = torch.zeros(case["points"], H.numel(), dtype=torch.complex128, device=DEV)
    if kind == "solve":
        n = parts[0].n
        state["Y"] = torch.randn(n, case["rhs"], generator=gen, device=DEV, dtype=torch.complex128)
        state["X"] = torch.zeros_like(state["Y"])
        state["factors"] = nd.ndsi_factor_poles(state["plan"], H, S, _points(case))
    if case.get("tune"):
        nd.ndsi_autotune(state["plan"], H, S, MU, case["kT"], case["poles"])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "mlp":
        state["params"].copy_(state["start"])
        loss = nd.ndsi_mlp_train(state["params"], state["X"], state["T"], case["samples"], case["steps"], 3e-3)
        return dict(params=state["params"], loss=loss)
    plan, H, S = state["plan"], state["H"], state["S"]
    if kind == "density":
        nd.ndsi_density(plan, H, S, MU, case["kT"], case["poles"], state["rho"], state["ne"])
        return dict(rho=state["rho"], ne=state["ne"])
    if kind == "share":
        b, e, m0 = state["share"]
        nd.ndsi_density_poles(plan, H, S, MU, case["kT"], case["poles"], b, e, m0, state["rho"], state["ne"])
        return dict(rho=state["rho"], ne=state["ne"])
    if kind == "energy":
        nd.ndsi_density_energy(plan, H, S, MU, case["kT"], case["poles"], state["rho"], state["e"], state["ne"])
        return dict(rho=state["rho"], e=state["e"], ne=state["ne"])
    if kind == "batched":
        ns = len(_parts(case))
        nd.ndsi_density_batched(plan, H, S, [MU - 0.01 * i for i in range(ns)], [case["kT"]] * ns, case["poles"],
                                state["rho"], state["ne"])
        return dict(rho=state["rho"], ne=state["ne"])
    if kind == "mu":
        n_e = _parts(case)[0].n / 2.0
        mu, ne, _ = nd.ndsi_find_mu(plan, H, S, case["kT"], case["poles"], n_e, state["rho"], tol_electrons=1e-10)
        return dict(rho=state["rho"], mu=mu, ne=ne)
    if kind == "green":
        f = nd.ndsi_factor_poles(plan, H, S, _points(case))
        nd.ndsi_selinv(f, state["G"])
        return state["G"]
    if kind == "dos":
        return nd.ndsi_dos(plan, H, S, _energies(case), case["eta"])
    if kind == "solve":
        return nd.ndsi_factors_solve(state["factors"], 0, state["Y"], state["X"])
    raise ValueError(kind)


@functools.lru_cache(maxsize=64)
def _cost(key):
    """Dense work per point and pattern size of a case's plan (host analysis only)."""
    case = dict(key)
    info = nd.ndsi_plan_info(_plan(case))
    return info["flops_per_pole"], info["nnz"], info["n"], info["front_elems"]


def work(case):
    kind = case["kind"]
    if kind == "mlp":
        macs = 32 * 64 + 64 * 64 + 64
        return dict(bytes=4.0 * (33 * case["samples"] + 2 * 6337), flops=6.0 * macs * case["samples"] * case["steps"])
    flops, nnz, n, front = _cost(tuple(sorted(case.items())))
    if kind == "solve":
        # lower triangles of the factors read once for all right-hand sides; A_J^{-1} and L_RJ used twice
        return dict(bytes=8.0 * front + 32.0 * n * case["rhs"], flops=8.0 * front * case["rhs"])
    points = {"density": lambda: case["poles"] + 1, "batched": lambda: case["poles"] + 1, "energy": lambda: case["poles"] + 4,
              "share": lambda: case["poles"] // case["world"] + 1, "green": lambda: case["points"],
              "dos": lambda: case["points"], "mu": lambda: 7 * (case["poles"] + 1)}[kind]()
    out = {"green": 16.0 * nnz * points, "energy": 16.0 * nnz, "dos": 8.0 * points}.get(kind, 8.0 * nnz)
    return dict(bytes=16.0 * nnz + out, flops=flops * points)


# -------------------------------------------------------------------------- 64-bit references ---
def _poles(M):
    """Poles and residues of the continued fraction of the Fermi function with M pole pairs."""
    k = np.arange(1, 2 * M)
    b = 1.0 / np.sqrt((2.0 * k - 1.0) * (2.0 * k + 1.0))
    lam, v = np.linalg.eigh(np.diag(b, 1) + np.diag(b, -1))
    keep = lam > 0
    lam, v1 = lam[keep][::-1], v[0, keep][::-1]
    return 2.0 / lam, -(v1 * v1) / (lam * lam)


def _dense(part, values):
    rows = torch.as_tensor(np.repeat(np.arange(part.n), np.diff(part.rowptr)), device=DEV)
    cols = torch.as_tensor(part.col.astype(np.int64), device=DEV)
    out = []
    for v in values:
        m = torch.zeros(part.n, part.n, dtype=torch.float64, device=DEV)
        m[rows, cols] = v
        out.append(m)
    return out, rows, cols


def _eigen(part, H, S):
    """Eigenpairs of H c = eps S c with C^T S C = 1, and the pattern's rows and columns."""
    (Hd, Sd), rows, cols = _dense(part, (H, S))
    L = torch.linalg.cholesky(Sd)
    A = torch.linalg.solve_triangular(L, Hd, upper=False)
    A = torch.linalg.solve_triangular(L, A.T.contiguous(), upper=False)
    eps, V = torch.linalg.eigh(0.5 * (A + A.T))
    return eps, torch.linalg.solve_triangular(L.T, V, upper=True), rows, cols


def _fermi(eps, mu, kT, M):
    z, R = _poles(M)
    f = torch.ones_like(eps)
    for zp, Rp in zip(z, R):
        y = zp * kT
        f += (-4.0 * Rp * kT) * (mu - eps) / ((mu - eps) ** 2 + y * y)
    return f


def _energy(eps, mu, kT, M):
    z, R = _poles(M)
    e = eps + 4.0 * kT * float(R.sum())
    for zp, Rp in zip(z, R):
        y = zp * kT
        d = (mu - eps) ** 2 + y * y
        e = e - 4.0 * kT * Rp * (mu * (mu - eps) + y * y) / d   # Re(alpha / (alpha - eps))
    return e


def _on_pattern(C, weight, rows, cols):
    return ((C * weight) @ C.T)[rows, cols]


def _exact_mlp(case, seed):
    params, X, T = _mlp_inputs(case, seed)
    x, t, n = X.double(), T.double(), case["samples"]
    p = params.double()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    b1, b2, lr, eps = float(np.float32(0.9)), float(np.float32(0.999)), float(np.float32(3e-3)), float(np.float32(1e-8))
    loss = 0.0
    for s in range(1, case["steps"] + 1):
        q = p.clone().requires_grad_(True)
        w1, c1, w2, c2, w3, c3 = torch.split(q, [2048, 64, 4096, 64, 64, 1])
        h = torch.tanh(torch.tanh(x @ w1.view(64, 32).T + c1) @ w2.view(64, 64).T + c2)
        err = ((h @ w3 + c3 - t) ** 2).sum() / n
        g, = torch.autograd.grad(err, q)
        loss = float(err.detach())
        m = b1 * m + (1 - b1) * g
        v = b2 * v + (1 - b2) * g * g
        p = p - lr * (m / (1 - b1 ** s)) / (torch.sqrt(v / (1 - b2 ** s)) + eps)
    return dict(params=p, loss=loss)


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _exact_mlp(case, seed)
    parts = _parts(case)
    if max(p.n for p in parts) > EXACT_MAX_N or sum(p.n ** 3 for p in parts) > 2.9e11:
        return None
    gen = _generator(seed)
    hs = [p.values(gen) for p in parts]
    if kind in ("green", "solve"):
        (Hd, Sd), rows, cols = _dense(parts[0], hs[0])
        if kind == "solve":
            Y = torch.randn(parts[0].n, case["rhs"], generator=gen, device=DEV, dtype=torch.complex128)
            return torch.linalg.solve(complex(_points(case)[0]) * Sd - Hd, Y)
        G = torch.empty(case["points"], rows.numel(), dtype=torch.complex128, device=DEV)
        for q, z in enumerate(_points(case)):
            G[q] = torch.linalg.inv(complex(z) * Sd - Hd)[rows, cols]
        return G
    if kind == "dos":
        eps = _eigen(parts[0], *hs[0])[0]
        E = torch.as_tensor(_energies(case), device=DEV)
        eta = case["eta"]
        return (2.0 / math.pi * eta / ((E[:, None] - eps[None, :]) ** 2 + eta * eta)).sum(1).cpu().numpy()
    rho, ne, en, mu_found = [], [], [], None
    for i, (part, (H, S)) in enumerate(zip(parts, hs)):
        eps, C, rows, cols = _eigen(part, H, S)
        mu, kT, M = MU - (0.01 * i if kind == "batched" else 0.0), case["kT"], case["poles"]
        if kind == "mu":
            lo, hi = float(eps.min()) - 1.0, float(eps.max()) + 1.0
            for _ in range(100):
                mu = 0.5 * (lo + hi)
                if float(_fermi(eps, mu, kT, M).sum()) < part.n / 2.0:
                    lo = mu
                else:
                    hi = mu
            mu_found = mu
        f = _fermi(eps, mu, kT, M)
        if kind == "share":
            b, e, m0 = nd.ndsi_pole_shard(M, case["rank"], case["world"])
            z, R = _poles(M)
            f = torch.full_like(eps, 1.0 if m0 else 0.0)
            for zp, Rp in zip(z[b:e], R[b:e]):
                y = zp * kT
                f += (-4.0 * Rp * kT) * (mu - eps) / ((mu - eps) ** 2 + y * y)
        rho.append(_on_pattern(C, f, rows, cols))
        ne.append(f.sum())
        if kind == "energy":
            en.append(_on_pattern(C, _energy(eps, mu, kT, M), rows, cols))
    out = dict(rho=torch.cat(rho), ne=torch.stack(ne))
    if kind == "energy":
        out["e"] = torch.cat(en)
    if kind == "mu":
        out["mu"], out["ne"] = mu_found, float(out["ne"][0])
    return out
