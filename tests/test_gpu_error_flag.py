"""What a kernel's wait leaves when it runs out (2: a staging copy, 3: a barrier of the persistent SAP) is reported by the call
that it happens in, as a CUDA error, and by no later one.  The flag is raised on the host: nothing waits.
"""
import numpy as np
import pytest

import synth
from cases import Case, THREE

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flag", [2, 3])
def test_a_timed_out_wait_is_reported_once(flag):
    import paper_1307_6101_gb300 as dd
    c = Case(**THREE)
    h = c.gpu(2)
    d, n, _ = h.level_info(0)
    dc, nc, _ = h.level_info(1)
    f = np.ascontiguousarray(synth.random_fields(1, d, n, 1))
    g = np.ascontiguousarray(synth.random_fields(1, dc, nc, 2))
    calls = {
        "apply": lambda: dd.ddamg_apply(h, 0, 1, f, np.zeros_like(f), 1),
        "smooth": lambda: dd.ddamg_smooth(h, 1, 1, g, g.copy(), 1, 1),
        "restrict": lambda: dd.ddamg_restrict(h, 0, 1, f, np.zeros_like(g), 1),
        "prolong": lambda: dd.ddamg_prolong(h, 0, 1, g, np.zeros_like(f), 1),
        "kcycle": lambda: dd.ddamg_kcycle(h, 0, 1, f, np.zeros_like(f), 1),
        "rebuild": lambda: dd.ddamg_rebuild(h, 0),
        "update_gauge": lambda: dd.ddamg_update_gauge(h, c.gauge(), 0),
        "solve": lambda: dd.ddamg_solve(h, f, np.zeros_like(f), 1, 1e-8),
    }
    for name, call in calls.items():
        assert dd.lib().ddamg_test_raise_flag(h.raw, flag) == 0
        with pytest.raises(dd.DdamgError) as e:
            call()
        assert e.value.code == -4 and "timed out" in str(e.value), (name, str(e.value))
        call()
