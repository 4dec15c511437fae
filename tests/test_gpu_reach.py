"""Closures with hub rows (more than 256 successors) on AUTO: the model by walks over the successor
lists where the closure is small, sweeps and squarings where it is not or its paths are long."""
import numpy as np
import pytest

import oracle
from paper_1608_00139_gb300 import inputs

pytestmark = pytest.mark.gpu


def relation(kind, n):
    rng = np.random.default_rng(n)
    e = inputs.pa_dag(n, n)
    if kind == "dag":  # hubs, few reachable constants per row
        pass
    elif kind == "cycles":  # small cycles: constants that reach themselves
        for i in rng.integers(0, n, 40):
            e[i, (i + 1) % n] = e[(i + 1) % n, i] = 1
        e[rng.integers(0, n, 30), rng.integers(0, n, 30)] = 1
    elif kind == "wide":  # one hub over everything else in two hops: frontiers wider than a warp's list
        e[:] = 0
        e[n - 1, : n // 2] = 1
        e[np.arange(n // 2), n // 2 + np.arange(n // 2) % (n // 2 - 1)] = 1
    elif kind == "dense":  # strongly connected around its hubs: not a small closure
        e |= e.T
    elif kind == "long":  # a hub at the head of a path longer than the walks go
        e[:] = 0
        order = rng.permutation(n)
        e[order[:-1], order[1:]] = 1
        e[order[0], order[:600]] = 1
    return e


@pytest.mark.parametrize("kind", ["dag", "cycles", "wide", "dense", "long"])
@pytest.mark.parametrize("n", [1025, 1279, 1280, 2047, 3100])
def test_hub_rows(ctx, n, kind):
    e = relation(kind, n)
    if e.sum(axis=1).max() <= 256:
        e[7, :300] = 1
    want = oracle.tc_model(e)
    for _ in range(2):  # the second call knows that the last one had hub rows
        bits, st = ctx.tc_closure(e)
        assert np.array_equal(bits, want)
        assert st["model_ones"] == int(np.unpackbits(want.view(np.uint8)).sum())
    packed, _ = ctx.tc_closure_bits(oracle.pack(e), n)
    assert np.array_equal(packed, want)
