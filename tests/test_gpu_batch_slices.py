"""GPU parity of the batch's column slices at the sizes where a slice, its successor lists or its
sweeps change hands: every model equals the oracle's bits (whole numbers: no tolerance)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1608_00139_gb300 import inputs

pytestmark = pytest.mark.gpu


def graph(n, degree, seed, loops=0.0):
    e = inputs.er_digraph(n, min(1.0, degree / max(n, 1)), seed)
    if loops:
        diag = np.random.default_rng(seed).random(n) < loops
        e[np.arange(n), np.arange(n)] = diag.astype(np.uint8)
    return e


def chain(n, length):
    e = np.zeros((n, n), dtype=np.uint8)
    at = np.arange(length - 1)
    e[at, at + 1] = 1
    return e


def half_chain(n, seed):
    """The last half of the constants a chain, the first half random: the slices of the first
    columns are done at once, the others are not."""
    e = graph(n, 3.0, seed)
    e[:, n // 2:] = 0
    e[n // 2:, :] = 0
    at = np.arange(n // 2, n - 1)
    e[at, at + 1] = 1
    return e


CASES = {
    # rows of 16, 8 and 4 words a slice, on both sides of each line, with a last partial slice
    "slice_edges": lambda: [graph(n, 2.0, 10 + k, 0.2) for k, n in
                            enumerate([1, 2, 63, 64, 65, 127, 129, 1023, 1024, 1025, 1153, 2047, 2048, 2049, 4096])],
    # one instance above the largest sliced one beside small ones
    "above_slices": lambda: [graph(4097, 1.5, 40), graph(100, 3.0, 41), graph(1500, 1.0, 42)],
    # successor lists that do not fit shared memory; complete relations; empty ones
    "dense": lambda: [graph(1000, 90.0, 50), np.ones((900, 900), np.uint8), np.zeros((1200, 1200), np.uint8),
                      graph(2000, 60.0, 51, 0.5)],
    # instances that go on to the batched rounds, with some of their slices done or none
    "handed_over": lambda: [chain(300, 300), half_chain(2000, 60), half_chain(1100, 61), chain(3000, 2500),
                            graph(700, 2.0, 62)],
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_batch_slices(ctx, name):
    gs = CASES[name]()
    dev = [torch.from_numpy(e).cuda() for e in gs]
    oracle.set_threads(0)
    ref = [oracle.tc_model(e) for e in gs]
    ones = sum(int(np.unpackbits(r.view(np.uint8)).sum()) for r in ref)
    for _ in range(2):  # the kept graph of the rounds the second time, other output buffers
        outs, st = ctx.tc_batch(dev)
        for e, b, r in zip(gs, outs, ref):
            assert np.array_equal(b.cpu().numpy().view(np.uint64), r), e.shape
        assert st["model_ones"] == ones
    outs, st = ctx.tc_batch(gs)  # host memory
    assert all(np.array_equal(b, r) for b, r in zip(outs, ref)) and st["model_ones"] == ones
