"""The product P^+ (term of D P) by column groups, and the orthonormalisation, at the sizes where the split of the
work changes: column counts around the groups of eight (FP32) and four (FP64) and the tiles of four, aggregates
that span a lattice direction (no hop leaves them), odd extents, and a second level (dof-contiguous fields).

The blocks against the oracle's: FP64 1e-12; FP32 products of the FP32-rounded operands 1e-5 (sums of up to some
hundred products with cancellation in the hop blocks).
"""
import numpy as np
import pytest

from cases import Case, rel

pytestmark = pytest.mark.gpu

CASES = [
    dict(dims=(4, 4, 4, 4), levels=2, agg=((2, 2, 2, 2),), n_tv=(1,), sap=((2, 2, 2, 2),)),
    dict(dims=(4, 4, 4, 8), levels=2, agg=((4, 2, 2, 4),), n_tv=(9,), sap=((2, 2, 2, 2),)),
    dict(dims=(6, 6, 6, 6), levels=2, agg=((3, 3, 3, 3),), n_tv=(17,), sap=((3, 3, 3, 3),)),
    dict(dims=(8, 8, 8, 8), levels=2, agg=((4, 4, 4, 4),), n_tv=(32,), sap=((4, 4, 4, 4),)),
    dict(dims=(8, 4, 4, 8), levels=3, agg=((2, 2, 2, 2), (2, 1, 2, 2)), n_tv=(5, 12), sap=((2, 2, 2, 2), (2, 2, 2, 2))),
]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c["dims"])) + "-" + "-".join(map(str, c["n_tv"])))
def test_coarse_operators_against_oracle(case, precision):
    import paper_1307_6101_gb300 as dd
    c = Case(**case)
    h, o = c.gpu(precision), c.oracle()
    for l in range(1, c.levels):
        d, n, _ = h.level_info(l)
        blk = np.zeros(tuple(d) + (9, n, n), dtype=np.complex128)
        dd.ddamg_get_coarse_operator(h, l, blk)
        st = o.levels[l].op
        ref = np.concatenate([st.diag[..., None, :, :], np.moveaxis(st.fwd, 0, -3), np.moveaxis(st.bwd, 0, -3)], -3)
        assert rel(blk, ref) <= (1e-12 if precision == 0 else 1e-5)
