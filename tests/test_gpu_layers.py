"""Same generation on the layers of an acyclic relation: the model and the real S~ against the
oracle at the edges of the route (one layer, the most layers it takes and one more, the most
parents per node it takes and one more, labels in any order, sizes around the words of a row)."""
import numpy as np
import pytest

import oracle
from paper_1608_00139_gb300 import dl

pytestmark = pytest.mark.gpu


def layered(n, levels, parents, seed):
    """A relation of exactly ``levels`` layers: a chain through them, every other node below some
    layer with 1 .. parents distinct parents in the layers above; labels permuted."""
    rng = np.random.default_rng(seed)
    level = np.concatenate([np.arange(levels), rng.integers(0, levels, n - levels)])
    p = np.zeros((n, n), np.uint8)
    for i in range(n):
        if level[i] == 0:
            continue
        if 1 <= i < levels:
            p[i, i - 1] = 1
        above = np.flatnonzero(level < level[i])
        k = min(int(rng.integers(1, parents + 1)), len(above)) - int(p[i].sum())
        if k > 0:
            p[i, rng.choice(above[p[i, above] == 0], k, replace=False)] = 1
    perm = rng.permutation(n)
    return p[np.ix_(perm, perm)]


CASES = [(1, 1, 1), (63, 1, 1), (64, 2, 1), (65, 9, 2), (130, 64, 3), (131, 65, 3), (257, 12, 4), (300, 12, 5),
         (333, 7, 16), (400, 7, 17), (1000, 20, 2)]


@pytest.mark.parametrize("n,levels,parents", CASES)
@pytest.mark.parametrize("with_b", [False, True])
def test_layers(ctx, n, levels, parents, with_b):
    p = layered(n, levels, parents, 7 * n + levels)
    b = (np.random.default_rng(n).random((n, n)) < 1.5 / n).astype(np.uint8) if with_b else None
    want = oracle.sg_model(p, b)
    bits, st = ctx.sg_least_model(p, b)
    assert np.array_equal(bits, want)
    assert st["model_ones"] == int(np.unpackbits(want.view(np.uint8)).sum())
    ref = oracle.sg_stilde_series(p, b)
    for path in ("auto", "fp64"):
        x, xb, sx = ctx.sg_real(p, b, path=path)
        # FP64 sums of at most 16 x 16 terms over at most 65 layers: well inside the FP64 paths' 1e-10
        assert np.abs(x - ref).max() <= 1e-12 * np.abs(ref).max()
        assert np.array_equal(xb, want)
        assert sx["model_ones"] == st["model_ones"]


def test_cycle_and_tiny_eps_leave_the_layers(ctx):
    """One edge back makes a cycle; with a tiny eps the entries of deep layers underflow and the
    model comes from the boolean route."""
    n = 200
    p = layered(n, 30, 2, 5)
    level = np.zeros(n, int)
    for _ in range(30):
        level = np.where(p.any(axis=1), 1 + (p * level[None, :]).max(axis=1), 0)
    deep = int(level.argmax())
    assert level[deep] == 29
    root = int(np.flatnonzero(p.sum(axis=1) == 0)[0])
    q = p.copy()
    q[root, deep] = 1
    assert np.array_equal(ctx.sg_least_model(q)[0], oracle.sg_model(q))
    x, bits, st = ctx.sg_real(p, eps=1e-30)
    assert np.array_equal(bits, oracle.sg_model(p))
    assert st["path_used"] == dl.PATHS["fp64"]
