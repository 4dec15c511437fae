"""R~2 of the transposed class on AUTO (FP32 correction series, FP64 residual) and by the FP64 series
against the oracle's series, at the edges of tiles and vectors, on relations whose series is fast, slow
(AUTO falls back to FP64) and empty, with hubs, self-loops and a smaller eps."""
import numpy as np
import pytest

import oracle  # noqa: F401
from oracle import transposed as tr
from paper_1608_00139_gb300 import dl, inputs

pytestmark = pytest.mark.gpu


def relation(kind, n):
    if kind == "er":
        return inputs.er_digraph(n, min(0.5, 3.0 / n), 9 + n, self_loops=True)
    if kind == "hub":
        return inputs.pa_dag(n, 5 + n)
    if kind == "complete":  # eps = 1/n: a slow series
        return (1 - np.eye(n)).astype(np.uint8)
    return np.zeros((n, n), np.uint8)


@pytest.mark.parametrize("kind,n", [("er", 1), ("er", 2), ("er", 3), ("er", 5), ("er", 63), ("er", 65), ("er", 255), ("er", 257),
                                    ("er", 1030), ("hub", 300), ("hub", 1025), ("complete", 24), ("complete", 40),
                                    ("empty", 70)])
def test_auto_and_fp64(ctx, kind, n):
    r1 = relation(kind, n)
    ref = tr.trans_rtilde_series(r1, tol=1e-19)
    want = tr.trans_model(r1)
    for path in ("auto", "fp64"):
        bits, st, x = ctx.transposed(r1, path=path, rtilde=True)
        assert np.array_equal(np.unpackbits(bits.view(np.uint8), axis=1, bitorder="little")[:, :n], want)
        # both stop at 1e-13 eps (a residual, a change); a contraction of 1 - 1/n multiplies it by n
        assert np.abs(x - ref).max() <= 1e-13 * max(10, 2 * n) * max(np.abs(ref).max(), 1e-300)
        assert st["final_resid"] <= 1e-13
        assert np.all(x[want == 0] == 0.0)  # (the oracle's series stops above the deepest entries)
        assert st["path_used"] == dl.PATHS["fp64"]
    eps = 0.25 * tr.trans_eps(r1)
    x = ctx.transposed(r1, eps=eps, rtilde=True)[2]
    ref = tr.trans_rtilde_series(r1, eps, tol=1e-19)
    assert np.abs(x - ref).max() <= 1e-12 * max(np.abs(ref).max(), 1e-300)
