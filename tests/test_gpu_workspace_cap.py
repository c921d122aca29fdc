"""max_workspace_bytes counts the basis scaling tables: the chunks of a sweep fit the cap beside them."""
import numpy as np
import pytest

from synth import lattice_system

pytestmark = pytest.mark.gpu


def test_scaling_tables_count():
    import torch
    import paper_1005_0088_gb300 as nd
    sysm = lattice_system((9, 8, 1), 3, "2d", 5)
    H, S = torch.as_tensor(sysm.H, device="cuda"), torch.as_tensor(sysm.S, device="cuda")
    rho = torch.zeros_like(H)
    M = 6

    def chunks(cap):
        """Chunks of a sweep over M poles and M0 under this cap; None when it is refused."""
        plan = nd.analyze_system(sysm, leaf_atoms=8, max_workspace_bytes=cap)
        nd.ndsi_profile_enable(plan, True)
        try:
            nd.ndsi_density(plan, H, S, -0.1, 0.02, M, rho)
        except nd.NdsiError as e:
            assert e.code == nd.ndsi.NDSI_ERR_OOM
            return None
        return nd.ndsi_profile_read(plan)["accumulate"]["launches"]

    def smallest(ok, lo, hi):
        while hi - lo > 1:
            mid = (lo + hi) // 2
            lo, hi = (lo, mid) if ok(mid) else (mid, hi)
        return hi

    top = 1 << 32
    one = smallest(lambda c: chunks(c) is not None, 1, top)    # bytes of one point
    whole = smallest(lambda c: chunks(c) == 1, one, top)       # the sweep in one chunk
    tables = 2 * sysm.nnz + 2 * sysm.n                         # the least they hold
    assert whole >= (M + 1) * one + tables, (whole, one, tables)
    assert chunks(one) == M + 1
