"""Single closures that go on in column slices after the speculative sweeps: sizes around the words of
a slice, graphs whose slices all finish, some or none, and the size where slices no longer fit.
Models equal the oracle's bits (whole numbers: no tolerance)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1608_00139_gb300 import inputs

pytestmark = pytest.mark.gpu


def half_chain(n, seed):
    e = inputs.er_digraph(n, 1.4 / n, seed)
    e[:, n // 2:] = 0
    e[n // 2:, :] = 0
    at = np.arange(n // 2, n - 1)
    e[at, at + 1] = 1
    return e


CASES = [("er", n, d) for n in (5249, 5377, 6000, 7937) for d in (1.2, 2.0)] + [
    ("half", 6001, 0), ("er", 10700, 1.5), ("er", 10800, 1.5)]


@pytest.mark.parametrize("kind,n,d", CASES)
def test_sparse_closures_above_one_fact_per_row(ctx, kind, n, d):
    oracle.set_threads(0)
    e = half_chain(n, n) if kind == "half" else inputs.er_digraph(n, d / n, n)
    e[n - 1, n - 1] = e[5, 5] = 1
    ref = oracle.tc_model(e)
    ones = int(np.unpackbits(ref.view(np.uint8)).sum())
    dev = torch.from_numpy(e).cuda()
    for _ in range(2):
        out, st = ctx.tc_closure(dev)[:2]
        assert np.array_equal(out.cpu().numpy().view(np.uint64), ref) and st["model_ones"] == ones
    out, st = ctx.tc_closure(e)[:2]
    assert np.array_equal(out, ref) and st["model_ones"] == ones


@pytest.mark.parametrize("n", [6081, 6144])
def test_output_aligned_to_its_words_only(ctx, n):
    """The model straight into a caller's output that starts 8 bytes into a buffer (rows of as many words
    as the workspace's: n in (np - 64, np]); the words around it stay as they were."""
    oracle.set_threads(0)
    e = inputs.er_digraph(n, 2.0 / n, n)
    ref = oracle.tc_model(e)
    w = ref.shape[1]
    buf = torch.full((n * w + 2,), -3, dtype=torch.int64, device="cuda")
    out = buf[1:1 + n * w].view(n, w)
    assert out.data_ptr() % 16 == 8
    _, st = ctx.tc_closure(torch.from_numpy(e).cuda(), out=out)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), ref)
    assert st["model_ones"] == int(np.unpackbits(ref.view(np.uint8)).sum())
    assert int(buf[0]) == -3 and int(buf[-1]) == -3


def test_sweep_counters_hold_sweeps_through_memory_only(ctx):
    """The steps that a slice takes in shared memory, and the walks of hub rows, are no sweep launches."""
    oracle.set_threads(0)
    n = 6000
    dev = torch.from_numpy(inputs.er_digraph(n, 2.5 / n, 1)).cuda()
    for _ in range(2):
        _, st = ctx.tc_closure(dev)
        assert 0 < st["sweep_launches"] < st["gpu_launches"] and st["recheck_sweeps"] > st["sweep_launches"]
    dag = inputs.pa_dag(3000, 3000)
    assert dag.sum(axis=1).max() > 256
    for _ in range(2):  # (the second call walks from the start)
        bits, st = ctx.tc_closure(dag)
        assert np.array_equal(bits, oracle.tc_model(dag))
    assert st["sweep_launches"] == 0 and st["ms_sweep"] == 0 and st["sweep_bytes"] == 0
