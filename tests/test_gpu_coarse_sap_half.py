"""Coarse SAP on FP16 blocks (a cluster per SAP block): against the oracle on the same FP16 data for each cluster size, rows
per warp of eight, four and two (dofs divisible by 8, 4 and 2), blocks that span a lattice direction (a neighbour in
both directions), 192 sites to a CTA (384-site blocks on two CTAs), and one to three right-hand sides (pairs and a
remainder).  FP32 bound: 2e-6 relative per sweep
pair; a column has the same bits alone and in a batch.
"""
import numpy as np
import pytest

import synth
from cases import Case, rel

pytestmark = pytest.mark.gpu

CASES = [
    (dict(dims=(8, 8, 8, 8), levels=3, agg=((2, 2, 2, 2), (2, 2, 2, 2)), n_tv=(12, 12), sap=((2, 2, 2, 2), (2, 2, 2, 2))),
     (16, 8, 4, 2)),
    (dict(dims=(8, 4, 8, 8), levels=3, agg=((2, 2, 2, 2), (2, 1, 2, 2)), n_tv=(10, 10), sap=((2, 2, 2, 2), (2, 2, 2, 2))),
     (16, 8)),
    (dict(dims=(8, 4, 4, 4), levels=3, agg=((2, 2, 2, 2), (2, 1, 1, 1)), n_tv=(5, 6), sap=((2, 2, 2, 2), (2, 2, 2, 2))),
     (16, 4, 2)),
    (dict(dims=(16, 8, 8, 12), levels=3, agg=((2, 2, 2, 2), (2, 2, 2, 2)), n_tv=(1, 1), sap=((2, 2, 2, 2), (4, 4, 4, 6))),
     (2, 16)),
]


@pytest.mark.parametrize("case,sizes", CASES, ids=["n24", "n20", "n10", "n2"])
def test_sweeps_against_oracle(case, sizes):
    import paper_1307_6101_gb300 as dd
    from oracle.precision import stencil_half
    from oracle.smoother import SAP
    c = Case(**case, max_rhs=3)
    h, o = c.gpu(0), c.oracle()      # FP64 products: the same FP16 data as the oracle's
    dd.ddamg_set_option(h, dd.DDAMG_OPT_HALF_STORAGE, 1)
    d, n, _ = h.level_info(1)
    sap = SAP(stencil_half(o.levels[1].op), c.sap[1], c.mr_steps)
    b = np.ascontiguousarray(synth.random_fields(3, d, n, 8))
    z0 = np.ascontiguousarray(synth.random_fields(3, d, n, 9))
    ref = [sap.smooth(b[r], z0[r], 1) for r in range(3)]
    for cls in sizes:
        dd.ddamg_set_option(h, dd.DDAMG_OPT_SAP_CLUSTER, cls)
        assert dd.ddamg_get_option(h, dd.DDAMG_OPT_SAP_CLUSTER) == cls
        dd.ddamg_set_option(h, dd.DDAMG_OPT_SAP_PERSIST, 0)
        z = z0.copy()
        dd.ddamg_smooth(h, 1, 1, b, z, 3, 1)
        for r in range(3):
            assert rel(z[r], ref[r]) <= 2e-6, (cls, r, rel(z[r], ref[r]))
        one = z0[2:].copy()
        dd.ddamg_smooth(h, 1, 1, b[2:].copy(), one, 1, 1)
        assert np.array_equal(one[0], z[2])
