"""Restriction, interpolation and field export at the sizes where their work split changes: column groups of four and
sixteen and their remainders, row tiles of four, odd aggregate volumes (no pairs of sites per thread), test vectors
from 1 to 32, and the second level (dof-contiguous fields, odd dofs per chirality).

Against the oracle: FP64 1e-12, FP32 on FP32 or FP16 storage 2e-6; a column has the same bits alone and in a batch.
"""
import numpy as np
import pytest

import synth
from cases import Case, rel

pytestmark = pytest.mark.gpu

CASES = [
    dict(dims=(4, 4, 4, 4), levels=2, agg=((2, 2, 2, 2),), n_tv=(1,), sap=((2, 2, 2, 2),)),
    dict(dims=(6, 6, 6, 6), levels=2, agg=((3, 3, 3, 3),), n_tv=(9,), sap=((3, 3, 3, 3),)),
    dict(dims=(8, 8, 4, 8), levels=2, agg=((4, 4, 4, 4),), n_tv=(32,), sap=((4, 4, 4, 4),)),
    dict(dims=(8, 4, 8, 8), levels=3, agg=((2, 2, 2, 2), (2, 1, 2, 2)), n_tv=(5, 7), sap=((2, 2, 2, 2), (2, 2, 2, 2))),
]


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c["dims"])) + "-" + "-".join(map(str, c["n_tv"])))
def test_transfers_against_oracle(case, precision):
    import paper_1307_6101_gb300 as dd
    from oracle.precision import interpolation_half
    from oracle.transfer import prolong, restrict
    c = Case(**case, max_rhs=1)
    h, o = c.gpu(precision), c.oracle()
    tol = 1e-12 if precision == 0 else 2e-6
    for l in range(c.levels - 1):
        d, n, _ = h.level_info(l)
        dc, nc, _ = h.level_info(l + 1)
        P = o.levels[l].P if precision < 2 else interpolation_half(o.levels[l].P, c.agg[l])
        for cols in (1, 5, 18):
            f = np.ascontiguousarray(synth.random_fields(cols, d, n, 3 + l))
            phi = np.ascontiguousarray(synth.random_fields(cols, dc, nc, 4 + l))
            fc, pf = np.zeros_like(phi), np.zeros_like(f)
            dd.ddamg_restrict(h, l, min(precision, 1), f, fc, cols)
            dd.ddamg_prolong(h, l, min(precision, 1), phi, pf, cols)
            for r in range(cols):
                assert rel(fc[r], restrict(P, c.agg[l], f[r])) <= tol
                assert rel(pf[r], prolong(P, c.agg[l], phi[r])) <= tol
            one, onef = np.zeros_like(phi[:1]), np.zeros_like(f[:1])
            dd.ddamg_restrict(h, l, min(precision, 1), f[-1:].copy(), one, 1)
            dd.ddamg_prolong(h, l, min(precision, 1), phi[-1:].copy(), onef, 1)
            assert np.array_equal(one[0], fc[-1]) and np.array_equal(onef[0], pf[-1])
