"""FP32 SAP on 2^4 blocks (half a warp per block): against the oracle on FP32 and FP16 storage.

Block counts that leave the last CTA partly empty, both directions of the antiperiodic sign (a lattice two blocks long in
time), and a lattice of extent 2 in one direction, which takes the general kernel.  Two sweeps of chained FP32
applications, each within 2e-6 relative.
"""
import numpy as np
import pytest

import synth
from cases import Case, rel

pytestmark = pytest.mark.gpu

LATTICES = [(4, 4, 4, 4), (4, 4, 4, 12), (8, 4, 12, 4), (4, 4, 2, 8)]


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("dims", LATTICES, ids=lambda v: "x".join(map(str, v)))
def test_b2_sweep_against_oracle(dims, precision):
    import paper_1307_6101_gb300 as dd
    from oracle.precision import fine_op_half
    from oracle.smoother import SAP
    b2 = (2, 2, 2, 2)
    c = Case(dims=dims, levels=2, agg=(b2,), n_tv=(2,), sap=(b2,), max_rhs=3)
    h, o = c.gpu(precision), c.oracle()
    op = o.levels[0].op if precision == 1 else fine_op_half(c.gauge(), c.m0, c.csw, c.bc_t)
    sap = SAP(op, b2, c.mr_steps)
    f = np.ascontiguousarray(synth.random_spinors(3, dims, 5))
    z = np.ascontiguousarray(synth.random_spinors(3, dims, 6))
    z1 = z.copy()
    dd.ddamg_smooth(h, 0, 1, f, z1, 3, 1)
    one = z[2:].copy()
    dd.ddamg_smooth(h, 0, 1, f[2:].copy(), one, 1, 1)
    assert np.array_equal(one[0], z1[2])      # a column alone and in a batch
    for r in range(3):
        assert rel(z1[r], sap.smooth(f[r], z[r], 1)) <= 2e-6
