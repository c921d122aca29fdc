"""Split-precision products at the edges of the tensor-core kernel's K blocks (32 complex), exact chunks
(128) and read-out periods (256 and 512), for every slice count and accumulator layout.

A system of three atoms in a row, two leaves of s orbitals around a separator of r: the schedule's
products are L = B A^{-1} (K = s), the Schur update (K = s) and T = G_RR L (K = r).

Tolerance: digits cut at 2^-(8 S - 1) of the row maximum leave a product error of about
2^-(8 S - 1) sqrt(2 K) relative to the row and column maxima, amplified by at most cond(X) <= 240
(spectral width 6 over 0.25 Im z at Im z = 0.1): with K <= 600, S = 6: 8e-15 * 35 * 240 = 7e-11, S = 5:
1.7e-8, S = 4: 4.4e-6.  The four-accumulator layout's tail floor is 2^-38 of the result: 3.6e-12 * 240 = 9e-10.
Twenty times these are asserted below 1 (a sum dropped or read twice is off by 2^-8 or more of a scale)."""
import numpy as np
import pytest

from oracle.dense import green_dense, on_pattern
from synth import csr_from_dense

pytestmark = pytest.mark.gpu

SPREAD = {4: 4.4e-6, 5: 1.7e-8, 6: 9e-10, 7: 9e-10}


def system(s, r, seed):
    rng = np.random.default_rng(seed)
    n = 2 * s + r
    a = rng.normal(0, 0.1 / np.sqrt(max(n / 64, 1)), (n, n))
    H = (a + a.T) / 2 + np.diag(rng.uniform(-1, 1, n))
    w = rng.uniform(-1, 1, (n, n))
    w = (w + w.T) / 2
    np.fill_diagonal(w, 0.0)
    S = np.eye(n) + min(0.05, 0.75 / float(np.abs(w).sum(1).max())) * w
    H[:s, s + r:] = H[s + r:, :s] = 0.0
    S[:s, s + r:] = S[s + r:, :s] = 0.0
    centers = np.array([[0.0, 0, 0], [1.0, 0, 0], [2.0, 0, 0]])
    return csr_from_dense(H, S, centers, np.repeat(np.arange(3, dtype=np.int32), [s, r, s]))


def check(s, r, **opts):
    import torch
    import paper_1005_0088_gb300 as nd
    sysm = system(s, r, 1000 * s + r)
    z = [-0.12 + 0.1j, 0.3 + 1.0j]
    plan = nd.analyze_system(sysm, leaf_atoms=1, precision=nd.NDSI_PREC_SPLIT, **opts)
    f = nd.ndsi_factor_poles(plan, torch.as_tensor(sysm.H, device="cuda"), torch.as_tensor(sysm.S, device="cuda"), np.array(z))
    G = torch.zeros((len(z), sysm.nnz, 2), dtype=torch.float64, device="cuda")
    nd.ndsi_selinv(f, G)
    g = G.cpu().numpy()
    g = g[..., 0] + 1j * g[..., 1]
    Hd, Sd = sysm.dense()
    err = 0.0
    for q, zq in enumerate(z):
        ref = on_pattern(green_dense(Hd, Sd, zq), sysm)
        err = max(err, float(np.max(np.abs(g[q] - ref)) / np.max(np.abs(ref))))
    assert err < 20 * SPREAD[opts.get("split_slices", 6)], err


@pytest.mark.parametrize("s,r", [(31, 33), (32, 128), (33, 129), (64, 255), (127, 257), (129, 384), (256, 40), (257, 41),
                                 (385, 79), (512, 17), (513, 130), (90, 600)])
def test_k_edges(s, r):
    check(s, r)


@pytest.mark.parametrize("slices", [4, 5, 6, 7])
@pytest.mark.parametrize("bands", [0, 4, 5])
def test_layouts(slices, bands):
    check(290, 161, split_slices=slices, split_bands=bands)
