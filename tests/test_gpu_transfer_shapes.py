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


@pytest.mark.parametrize("side,n_tv,bound", [(4, 20, 1.11e-7), (4, 32, 1.15e-7), (6, 12, 1.79e-7)])
def test_single_column_rounding(side, n_tv, bound):
    """Restriction of one column from FP16 storage on side^4 aggregates: not further from 64 bits than with a lane per site
    and a butterfly over the lanes.  A rounding to FP32 is off by 2^-24 / sqrt(3) = 3.4e-8 of the value rounded (rms), and a
    chain of k sums of like terms by k / 2 such errors of its result, independently of other chains.  With 6 side^4 products
    of two FMAs per real part: 12 FMAs per site, sites / 256 of them in a lane's chain, five sums in the butterfly, eight
    warps in a chain, the scale and the rounding of the field make the error 3.4e-8 sqrt(6 + 5 + 4 + 1 + 1) = 1.4e-7 for
    side 4 if every lane's sum were of the size of the result; 1.11e-7 emulated, and 1.79e-7 measured for side 6.  Chains
    of three chunks per lane gave 1.33e-7 (side 4, 20 test vectors).  32 test vectors: 1.15e-7, since the 2560 values and four
    fields leave about 1 % of noise.
    """
    import paper_1307_6101_gb300 as dd
    from oracle.precision import interpolation_half
    from oracle.transfer import restrict
    agg = (side,) * 4
    c = Case(dims=(16, 8, 8, 8) if side == 4 else (12, 12, 6, 6), levels=2, agg=(agg,), n_tv=(n_tv,), sap=((2, 2, 2, 2),))
    h, o = c.gpu(0), c.oracle()
    dd.ddamg_set_option(h, dd.DDAMG_OPT_HALF_STORAGE, 1)
    dd.ddamg_set_option(h, dd.DDAMG_OPT_COARSE_TC, 0)      # the kernel for one right-hand side
    d, n, _ = h.level_info(0)
    dc, nc, _ = h.level_info(1)
    P = interpolation_half(o.levels[0].P, agg)
    err = []
    for seed in range(4):
        f = np.ascontiguousarray(synth.random_fields(1, d, n, 3 + seed))
        fc = np.zeros((1,) + tuple(dc) + (nc,), dtype=complex)
        dd.ddamg_restrict(h, 0, 1, f, fc, 1)
        err.append(rel(fc[0], restrict(P, agg, f[0])))
    assert np.mean(err) <= bound, err


@pytest.mark.parametrize("precision", [1, 2])
def test_overflow_stays_infinite(precision):
    """An entry beyond the FP32 range makes its aggregate's sums of that chirality infinite, not NaN, and no others."""
    import paper_1307_6101_gb300 as dd
    c = Case(dims=(8, 8, 4, 4), levels=2, agg=((4, 4, 4, 4),), n_tv=(5,), sap=((4, 4, 4, 4),))
    h = c.gpu(precision)
    d, n, _ = h.level_info(0)
    dc, nc, _ = h.level_info(1)
    f = np.ascontiguousarray(synth.random_fields(1, d, n, 3))
    ref, fc = np.zeros((2, 1) + tuple(dc) + (nc,), dtype=complex)
    dd.ddamg_restrict(h, 0, 1, f, ref, 1)
    f[0, 1, 1, 1, 1, 0] = 1e300
    dd.ddamg_restrict(h, 0, 1, f, fc, 1)
    hit = np.zeros(fc.shape, dtype=bool)
    hit[0, 0, 0, 0, 0, :5] = True
    assert np.isinf(fc[hit].real).all() and np.isinf(fc[hit].imag).all()
    assert np.array_equal(fc[~hit], ref[~hit])
