"""FP64-path products in 57-bit fixed point: widths around the tile, pivot and chunk sizes, basis
functions of very different scale, and non-finite input.

Tolerances: the kernels are backward stable to a small multiple of u = 2^-53 times the order of the
block, so G = X^{-1} is accurate to about n u cond(X) relative to its largest element; the shifts below
give cond(X) <= (spectral width 6) / (0.25 Im z), n <= 400, so 4e2 * 1.1e-16 * 240 = 1.1e-11 at
Im z = 0.1 and 1e-11 is asserted (the other tests of the same entry points assert 1e-11 as well).
Scaling the basis by powers of two changes no rounding (launch_basis_scale takes it out exactly);
the same tolerance is asserted."""
import numpy as np
import pytest

from oracle.dense import green_dense, on_pattern
from synth import csr_from_dense, lattice_system

pytestmark = pytest.mark.gpu

TOL = 1e-11


def lib():
    import paper_1005_0088_gb300 as nd
    nd.load()
    return nd


def selected_inverse(sysm, z, **opts):
    import torch
    nd = lib()
    plan = nd.analyze_system(sysm, **opts)
    nd.ndsi_plan_check(plan)
    H = torch.as_tensor(sysm.H, device="cuda")
    S = torch.as_tensor(sysm.S, device="cuda")
    f = nd.ndsi_factor_poles(plan, H, S, np.asarray(z))
    G = torch.zeros((len(z), sysm.nnz, 2), dtype=torch.float64, device="cuda")
    nd.ndsi_selinv(f, G)
    g = G.cpu().numpy()
    return g[..., 0] + 1j * g[..., 1]


def worst(sysm, z, g):
    Hd, Sd = sysm.dense()
    err = 0.0
    for q, zq in enumerate(z):
        ref = on_pattern(green_dense(Hd, Sd, zq), sysm)
        err = max(err, float(np.max(np.abs(g[q] - ref)) / np.max(np.abs(ref))))
    return err


Z = [-0.12 + 0.1j, 0.4 + 1.0j, 1e7j]


# one supernode of n columns: the diagonal-block kernel alone, at the edges of its 8 x 8 blocks, 16-wide
# pivots and width classes (64, 80, 128 columns), and past one outer block
@pytest.mark.parametrize("n", [1, 7, 8, 9, 15, 16, 17, 24, 31, 33, 63, 64, 65, 79, 80, 81, 96, 120, 127, 128, 129, 145, 257])
def test_single_block_widths(n):
    rng = np.random.default_rng(n)
    a = rng.normal(0, 0.1, (n, n))
    H = (a + a.T) / 2 + np.diag(rng.uniform(-1, 1, n))
    w = rng.uniform(-1, 1, (n, n))
    w = (w + w.T) / 2
    np.fill_diagonal(w, 0.0)
    S = np.eye(n) + min(0.05, 0.75 / max(float(np.abs(w).sum(1).max()), 1e-300)) * w
    sysm = csr_from_dense(H, S)
    sysm.atom_of_basis[:] = 0
    sysm.centers = np.zeros((1, 3))
    assert worst(sysm, Z, selected_inverse(sysm, Z)) < TOL


# several fronts: panel, update and selected-inverse products of ragged widths, K around 16 and 32
@pytest.mark.parametrize("shape,orb,kind,leaf", [((40, 1, 1), 1, "1d", 4), ((33, 1, 1), 7, "1d", 5), ((11, 7, 1), 3, "2d", 9),
                                                 ((9, 8, 1), 5, "2d", 12), ((5, 4, 3), 3, "3d", 8), ((6, 5, 4), 2, "3d", 31)])
def test_ragged_fronts(shape, orb, kind, leaf):
    sysm = lattice_system(shape, orb, kind, 909)
    assert worst(sysm, Z, selected_inverse(sysm, Z, leaf_atoms=leaf)) < TOL


# basis functions scaled by powers of two over 2^+-20: X -> D X D, G -> D^-1 G D^-1, exactly
@pytest.mark.parametrize("shape,orb,kind", [((40, 1, 1), 4, "1d"), ((8, 7, 1), 4, "2d")])
def test_scaled_basis(shape, orb, kind):
    sysm = lattice_system(shape, orb, kind, 77)
    z = Z[:2]
    d = 2.0 ** np.random.default_rng(5).integers(-20, 21, sysm.n)
    rows = sysm.rows()
    sc = d[rows] * d[sysm.col]
    ref = selected_inverse(sysm, z, leaf_atoms=10)
    sysm.H, sysm.S = sysm.H * sc, sysm.S * sc
    g = selected_inverse(sysm, z, leaf_atoms=10) * sc
    assert float(np.max(np.abs(g - ref)) / np.max(np.abs(ref))) < TOL


def test_non_finite_input_is_reported():
    nd = lib()
    for bad in (np.inf, np.nan):
        sysm = lattice_system((6, 5, 1), 3, "2d", 4)
        sysm.H[sysm.nnz // 2] = bad
        with pytest.raises(nd.NdsiError) as ei:
            selected_inverse(sysm, Z[:1], leaf_atoms=8)
        assert ei.value.code == nd.ndsi.NDSI_ERR_SINGULAR
