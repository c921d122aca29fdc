"""FP64-path GEMMs with inner sizes at the edges of their chunks of 64 and of the 16-wide pivots.

A system of three atoms in a row, two leaves of s orbitals around a separator of r: L = B A^{-1} and the Schur update have
K = s, T = G_RR L and G_JJ = A^{-1} + L^T T have K = r.  H has entries N(0, 1/n) and S = I: the spectrum is within [-2, 2]
and cond(z S - H) <= 4 at Im z = 0.7, so 20 sqrt(n) u cond of the largest element is allowed (4e-14 .. 2e-13); a chunk
left out is off by 1e-2 or more."""
import numpy as np
import pytest

from tests.test_gpu_split_scales import U, Z, matrices
from synth import csr_from_dense

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,r", [(63, 64), (64, 65), (65, 63), (127, 128), (128, 129), (129, 127), (191, 33), (192, 193),
                                 (193, 1), (1, 257), (17, 320)])
def test_inner_sizes(s, r):
    import torch
    import paper_1005_0088_gb300 as nd
    H, X = matrices(s, r)
    n = 2 * s + r
    centers = np.array([[0.0, 0, 0], [1.0, 0, 0], [2.0, 0, 0]])
    sysm = csr_from_dense(H, np.eye(n), centers, np.repeat(np.arange(3, dtype=np.int32), [s, r, s]))
    plan = nd.analyze_system(sysm, leaf_atoms=1)
    nd.ndsi_plan_check(plan)
    f = nd.ndsi_factor_poles(plan, torch.as_tensor(sysm.H, device="cuda"), torch.as_tensor(sysm.S, device="cuda"), np.array([Z]))
    G = torch.zeros((1, sysm.nnz, 2), dtype=torch.float64, device="cuda")
    nd.ndsi_selinv(f, G)
    g = G.cpu().numpy()[0]
    err = np.max(np.abs(g[:, 0] + 1j * g[:, 1] - X[sysm.rows(), sysm.col])) / np.max(np.abs(X))
    assert err < 20 * np.sqrt(n) * U * np.linalg.cond(X), err
