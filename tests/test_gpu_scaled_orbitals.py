"""FP64-path results for a normalised basis (S_ii = 1) whose on-site energies and couplings span many decades:
core levels of 10^2 to 10^10 among valence orbitals of order 1, and energies spread evenly over 12 decades.

Reference: the inverse of z S - H, refined once by Newton's step in long double (64 bits of mantissa or more).
Tolerance: an elimination that keeps every element's bits is backward stable in the basis scaled by
d_i = (|H_ii| + |z|)^-1/2, so the error of G_ij / (d_i d_j) is about n u cond(D X D) of its largest element,
with u = 2^-53.  That is asserted (cond computed from the scaled matrix); the whole of G is held to it, not
only its largest elements.  Products exact relative to a row's maximum, without a scaling that brings the
orbitals together, miss it by 10^2 to 10^5 for all but the smallest range."""
import numpy as np
import pytest

from synth import lattice_system

pytestmark = pytest.mark.gpu

Z = np.array([-0.12 + 0.1j, 0.4 + 1.0j, 0.3 + 30j, 3e3j])


def heavy(sysm, size, seed):
    """S = I; every fifth orbital at -size with couplings of its 0.4th power."""
    rng = np.random.default_rng(seed)
    rows, col = sysm.rows(), sysm.col
    sysm.S = (rows == col).astype(float)
    core = np.zeros(sysm.n, bool)
    core[rng.permutation(sysm.n)[: sysm.n // 5]] = True
    off = rows != col
    H = sysm.H.copy()
    H[(core[rows] | core[col]) & off] *= 10 * size ** 0.4
    diag = ~off & core[rows]
    H[diag] = -size * rng.uniform(0.5, 2.0, int(diag.sum()))
    sysm.H = H
    return sysm


def spread(sysm, size, seed):
    """S = I; H scaled by the square roots of energies spread evenly over the logarithm of `size`."""
    rng = np.random.default_rng(seed)
    rows, col = sysm.rows(), sysm.col
    sysm.S = (rows == col).astype(float)
    d = size ** rng.uniform(0.0, 0.5, sysm.n)
    sysm.H = sysm.H * d[rows] * d[col]
    return sysm


SYSTEMS = {"core_1e4": lambda: heavy(lattice_system((8, 6, 1), 3, "2d", 31), 1e4, 1),
           "core_1e10": lambda: heavy(lattice_system((8, 6, 1), 3, "2d", 32), 1e10, 2),
           "core_1e10_box": lambda: heavy(lattice_system((4, 4, 3), 3, "3d", 33), 1e10, 3),
           "spread_1e12": lambda: spread(lattice_system((40, 1, 1), 4, "1d", 34), 1e12, 4)}


def exact(sysm, z):
    Hd, Sd = sysm.dense()
    A = z * Sd - Hd
    d = 1.0 / np.sqrt(np.abs(np.diag(Hd)) + abs(z))
    B = A * d[:, None] * d[None, :]
    X = np.linalg.inv(B).astype(np.clongdouble)
    Bl = B.astype(np.clongdouble)
    X = X + X @ (np.eye(sysm.n, dtype=np.clongdouble) - Bl @ X)
    return X, d, sysm.n * 2.0 ** -53 * float(np.linalg.cond(B)) * float(np.max(np.abs(X)))


@pytest.mark.parametrize("name", SYSTEMS)
def test_orbitals_of_very_different_energy(name):
    import torch
    import paper_1005_0088_gb300 as nd
    sysm = SYSTEMS[name]()
    rows, col = sysm.rows(), sysm.col
    plan = nd.analyze_system(sysm, leaf_atoms=8)
    H, S = torch.as_tensor(sysm.H, device="cuda"), torch.as_tensor(sysm.S, device="cuda")
    f = nd.ndsi_factor_poles(plan, H, S, Z)
    k = 9
    rng = np.random.default_rng(7)
    Y = rng.normal(size=(sysm.n, k)) + 1j * rng.normal(size=(sysm.n, k))
    Xs = []
    for q in range(len(Z)):
        x = torch.zeros(sysm.n, k, dtype=torch.complex128, device="cuda")
        nd.ndsi_factors_solve(f, q, torch.as_tensor(Y, device="cuda"), x)
        Xs.append(x.cpu().numpy())
    G = torch.zeros((len(Z), sysm.nnz, 2), dtype=torch.float64, device="cuda")
    nd.ndsi_selinv(f, G)
    g = G.cpu().numpy()
    g = g[..., 0] + 1j * g[..., 1]
    D = nd.ndsi_dos(plan, H, S, np.array([-0.12]), 0.1)
    for q, z in enumerate(Z):
        X, d, tol = exact(sysm, complex(z))
        err = float(np.max(np.abs(g[q] / (d[rows] * d[col]) - X[rows, col])))
        assert err < tol, (name, z, "G", err, tol)
        # X Y in the scaled basis: the columns' sizes come in
        want = X @ (d[:, None] * Y)
        err = float(np.max(np.abs(Xs[q] / d[:, None] - want)))
        assert err < tol * float(np.max(np.sum(np.abs(d[:, None] * Y), axis=0))), (name, z, "solve", err)
        if q == 0:
            tr = -2.0 / np.pi * np.sum((X[rows, col] * d[rows] * d[col]).imag * sysm.S)
            assert abs(D[0] - float(tr)) < tol * float(np.sum(d * d)), (name, "dos")


def test_one_pole_of_the_density():
    """rho and Tr(rho S) of a single pole of the sum, 2 Re of its weighted G."""
    import torch
    import paper_1005_0088_gb300 as nd
    from oracle.poles import cf_poles
    sysm = SYSTEMS["core_1e10"]()
    rows, col = sysm.rows(), sysm.col
    mu, kT, M = -0.12, 0.05, 20
    zp, Rp = cf_poles(M)
    plan = nd.analyze_system(sysm, leaf_atoms=8)
    H, S = torch.as_tensor(sysm.H, device="cuda"), torch.as_tensor(sysm.S, device="cuda")
    rho = torch.zeros(sysm.nnz, dtype=torch.float64, device="cuda")
    ne = torch.zeros(1, dtype=torch.float64, device="cuda")
    nd.ndsi_density_poles(plan, H, S, mu, kT, M, 0, 1, False, rho, ne)
    X, d, tol = exact(sysm, mu + 1j * zp[0] * kT)
    w = -4.0 * Rp[0] * kT
    want = w * X[rows, col].real
    err = float(np.max(np.abs(rho.cpu().numpy() / (d[rows] * d[col]) - want)))
    assert err < abs(w) * tol, (err, abs(w) * tol)
    tr = float(np.sum(want * d[rows] * d[col] * sysm.S))
    assert abs(float(ne.cpu()[0]) - tr) < abs(w) * tol * float(np.sum(d * d))


def test_systems_of_a_batch_are_scaled_by_themselves():
    """A plain system beside one with core levels has the bits it has beside its like (same shapes, so the
    same schedule)."""
    import torch
    import paper_1005_0088_gb300 as nd
    plain = lattice_system((7, 5, 1), 3, "2d", 35)
    other = heavy(lattice_system((7, 5, 1), 3, "2d", 36), 1e10, 5)
    H = torch.as_tensor(np.concatenate([plain.H, other.H]), device="cuda")
    S = torch.as_tensor(np.concatenate([plain.S, other.S]), device="cuda")
    out = []
    for systems in ([plain, plain], [plain, other]):
        plan = nd.analyze_batched(systems, leaf_atoms=8)
        h, s = (H, S) if systems[1] is other else (torch.cat([H[: plain.nnz]] * 2), torch.cat([S[: plain.nnz]] * 2))
        rho = torch.zeros_like(h)
        ne = torch.zeros(2, dtype=torch.float64, device="cuda")
        nd.ndsi_density_batched(plan, h, s, [-0.12, -0.1], [0.02, 0.02], 20, rho, ne)
        out.append(rho[: plain.nnz].cpu().numpy())
    assert np.array_equal(out[0], out[1])
