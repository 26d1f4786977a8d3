"""FP64 fine-level kernels with six threads per site: the operator and SAP against the oracle.

The SAP cases cover each way a block is shared out: one CTA (2^4, with and without a partial last warp),
clusters whose last CTA is not full (3^4: 81 sites), clusters of eight (4^4, and 4x4x4x6 = 384 sites on few
blocks), blocks that span a lattice direction (hops that wrap inside, with the antiperiodic sign), and extents
1 and 2.  FP64 bound: 1e-12 relative per application, three chained applications here.
"""
import numpy as np
import pytest

import synth
from cases import Case, rel

pytestmark = pytest.mark.gpu

# dims, aggregate = SAP block
BLOCKS = [
    ((4, 4, 4, 4), (2, 2, 2, 2)),
    ((6, 6, 6, 12), (3, 3, 3, 3)),
    ((4, 8, 4, 8), (4, 4, 4, 4)),
    ((8, 8, 8, 8), (4, 4, 4, 4)),
    ((4, 4, 8, 12), (4, 4, 4, 6)),
    ((2, 4, 6, 4), (2, 1, 3, 2)),
    ((4, 4, 4, 6), (2, 2, 1, 3)),
]


@pytest.mark.parametrize("dims,block", BLOCKS, ids=lambda v: "x".join(map(str, v)))
def test_split_operator_and_sap_against_oracle(dims, block):
    import paper_1307_6101_gb300 as dd
    c = Case(dims=dims, levels=2, agg=(block,), n_tv=(1,), sap=(block,), max_rhs=2)
    h, o = c.gpu(0), c.oracle()
    f = np.ascontiguousarray(synth.random_spinors(2, dims, 5))
    z = np.ascontiguousarray(synth.random_spinors(2, dims, 6))
    out = np.zeros_like(f)
    dd.ddamg_apply(h, 0, 0, f, out, 2)
    z1 = z.copy()
    dd.ddamg_smooth(h, 0, 0, f, z1, 2, 1)
    one = z[:1].copy()
    dd.ddamg_smooth(h, 0, 0, f[:1].copy(), one, 1, 1)
    assert np.array_equal(one, z1[:1])      # a column alone and in a batch
    for r in range(2):
        assert rel(out[r], o.levels[0].op.apply(f[r])) <= 1e-12
        assert rel(z1[r], o.levels[0].sap.smooth(f[r], z[r], 1)) <= 1e-12


@pytest.mark.parametrize("dims,block,max_rhs", [((16, 8, 8, 8), (4, 4, 4, 4), 1), ((16, 8, 8, 8), (4, 4, 4, 4), 8),
                                                ((16, 8, 8, 8), (4, 4, 4, 4), 12), ((6, 6, 6, 4), (3, 3, 3, 2), 64)])
def test_sap_kernel_of_the_handles_batch(dims, block, max_rhs):
    """16 blocks of 4^4 sites per colour: six threads per site for batches of one and twelve, one thread per site for eight;
    8 blocks of 54 sites, four to a CTA: one thread per site for a batch of 64.  A column has the same bits alone and in a
    batch of any size."""
    import paper_1307_6101_gb300 as dd
    c = Case(dims=dims, levels=2, agg=(block,), n_tv=(1,), sap=(block,), max_rhs=max_rhs)
    h, o = c.gpu(0), c.oracle()
    f = np.ascontiguousarray(synth.random_spinors(9, dims, 5))
    z = np.ascontiguousarray(synth.random_spinors(9, dims, 6))
    z1, one = z.copy(), z[8:].copy()
    dd.ddamg_smooth(h, 0, 0, f, z1, 9, 1)
    dd.ddamg_smooth(h, 0, 0, f[8:].copy(), one, 1, 1)
    assert np.array_equal(one[0], z1[8])
    for r in (0, 8):
        assert rel(z1[r], o.levels[0].sap.smooth(f[r], z[r], 1)) <= 1e-12
