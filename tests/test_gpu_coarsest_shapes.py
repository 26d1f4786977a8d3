"""Coarsest odd-even GMRES on a thread-block cluster, a fixed number of steps (two cycles of m) against the oracle's:
one site of each parity per CTA and several, dofs divisible by 8, by 4 and by 2 only, the largest of the variant that
keeps its operator on chip, a single step per cycle, and a column's bits alone and in a batch.

FP64 1e-9 (as for the solve to tolerance).  FP32 on FP16 blocks 1e-4: up to ten steps, each off by at most n products
of 6e-8 relative to operands of order one, of an operator whose condition is below ten.
"""
import numpy as np
import pytest

import synth
from cases import Case, rel

pytestmark = pytest.mark.gpu

CASES = {
    "16x16": dict(dims=(8, 8, 8, 8), levels=2, agg=((4, 4, 4, 4),), n_tv=(8,), sap=((4, 4, 4, 4),)),
    "16x10": dict(dims=(4, 4, 4, 8), levels=2, agg=((2, 2, 2, 4),), n_tv=(5,), sap=((2, 2, 2, 4),)),
    "32x56": dict(dims=(8, 4, 4, 8), levels=2, agg=((2, 2, 2, 2),), n_tv=(28,), sap=((2, 2, 2, 2),)),
    "256x6": dict(dims=(8, 8, 8, 8), levels=2, agg=((2, 2, 2, 2),), n_tv=(3,), sap=((4, 4, 4, 4),)),
}


@pytest.mark.parametrize("m", [1, 5])
@pytest.mark.parametrize("name", CASES)
def test_fixed_steps_against_oracle(name, m):
    import paper_1307_6101_gb300 as dd
    from oracle.krylov import coarsest_solve
    from oracle.precision import even_odd_half
    c = Case(**CASES[name], m0=0.2, max_rhs=3, coarse_restart=m, extra=dict(coarse_tol=1e-14, coarse_cycles=2))
    h, o = c.gpu(0), c.oracle()
    dims, n, _ = h.level_info(1)
    b = np.ascontiguousarray(synth.random_fields(3, dims, n, 60))
    for half in (0, 1):
        if half:
            dd.ddamg_set_option(h, dd.DDAMG_OPT_HALF_STORAGE, 1)
        eo = even_odd_half(o.levels[1].op) if half else o.levels[1].eo
        z = np.zeros_like(b)
        dd.ddamg_coarse_solve(h, half, b, z, 3)
        for i in range(3):
            ref = coarsest_solve(eo, b[i], 1e-14, m, 2)[0]
            assert rel(z[i], ref) <= (1e-4 if half else 1e-9), (half, i, rel(z[i], ref))
        one = np.zeros_like(b[2:])
        dd.ddamg_coarse_solve(h, half, b[2:].copy(), one, 1)
        assert np.array_equal(one[0], z[2])
