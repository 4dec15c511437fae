"""The plain FP64 path at the edges of its 32 x 32 blocks, of its padding to 64 and of its two forms
(Gauss-Jordan up to 1024, elimination with a backward pass beyond): R~ against the oracle's LU."""
import numpy as np
import pytest

import oracle
from paper_1608_00139_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 96, 127, 129, 1023, 1024, 1025, 1089])
def test_blocks(ctx, n):
    e = inputs.er_digraph(n, min(0.5, 6.0 / max(n, 1)), 40 + n, self_loops=True)
    bits, st, x = ctx.tc_closure(e, path="fp64", rtilde=True)
    ref = oracle.tc_rtilde_lu(e, st["eps_used"])
    # the bound stated for the FP64 path
    assert np.abs(x - ref).max() <= 1e-10 * max(np.abs(ref).max(), 1e-300)
    assert np.array_equal(bits, oracle.tc_model(e))
    assert st["rows_rechecked"] == 0 and st["guard_flagged"] == 0
