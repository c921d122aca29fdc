"""Pivots whose squared modulus is subnormal (|p| from 0.8e-154 to 1.4e-154) are inverted, as every other non-zero one,
in the warp kernel (8 columns) and in the diagonal-block kernel (40 and 129 columns); a zero pivot is refused.

z S - H is 2^-512 times a well-conditioned matrix, so G is 2^512 times its inverse.  The subnormal numbers that come
up, |p|^2 and products of that size, are off by 2^-1074, 3e-16 of |p|^2 or less: the error is the usual n u cond of the
largest element, with cond <= 3 and n <= 129 below 5e-14; 1e-12 is asserted."""
import numpy as np
import pytest

from synth import csr_from_dense

pytestmark = pytest.mark.gpu

TINY = 2.0 ** -512      # 7.5e-155


def single_node(H, S):
    sysm = csr_from_dense(H, S)
    sysm.atom_of_basis[:] = 0
    sysm.centers = np.zeros((1, 3))
    return sysm


def green(sysm, z):
    import torch
    import paper_1005_0088_gb300 as nd
    plan = nd.analyze_system(sysm)
    f = nd.ndsi_factor_poles(plan, torch.as_tensor(sysm.H, device="cuda"), torch.as_tensor(sysm.S, device="cuda"),
                             np.array([z]))
    G = torch.zeros((1, sysm.nnz, 2), dtype=torch.float64, device="cuda")
    nd.ndsi_selinv(f, G)
    g = G.cpu().numpy()[0]
    return g[:, 0] + 1j * g[:, 1]


@pytest.mark.parametrize("n", [8, 40, 129])
def test_subnormal_squared_pivots(n):
    rng = np.random.default_rng(n)
    a = rng.normal(0, 0.1 / np.sqrt(n), (n, n))
    H = (a + a.T) / 2 + np.diag(rng.uniform(-0.1, 0.1, n))
    z = 1.0 + 1.0j                                     # every pivot near 1.4
    B = z * np.eye(n) - H
    sysm = single_node(H * TINY, np.eye(n))
    g = green(sysm, z * TINY)
    want = np.linalg.inv(B)[sysm.rows(), sysm.col]
    assert np.max(np.abs(g * TINY - want)) < 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("n", [8, 40])
def test_zero_pivot_is_refused(n):
    import paper_1005_0088_gb300 as nd
    H = np.diag(np.linspace(1.0, 2.0, n))
    H[3, 3] = 0.0
    with pytest.raises(nd.NdsiError) as e:
        green(single_node(H, np.eye(n)), 0.0)
    assert e.value.code == nd.ndsi.NDSI_ERR_SINGULAR
