"""The one-launch closure (AUTO up to n = 1024; 1025 and up take the general route) against the oracle: sizes at the edges of words, of the
16-column pieces of the ingest and of the CTAs' rows; sparse, dense, saturated and empty relations, rows
longer than a list, paths that need the squarings; bytes at any alignment and packed rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_1608_00139_gb300 import dl, inputs

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 15, 16, 17, 63, 64, 65, 127, 128, 129, 257, 511, 512, 513, 1000, 1023, 1024, 1025]


def relation(kind, n):
    rng = np.random.default_rng(n)
    if kind == "sparse":
        return inputs.er_digraph(n, min(1.0, 2.5 / n), n + 3, self_loops=True)
    if kind == "dense":
        return inputs.er_digraph(n, 0.2, n + 4)
    if kind == "idle":  # a fifth of the constants without facts, rows of some 40 successors
        e = inputs.er_digraph(n, min(1.0, 40.0 / n), n + 5)
        off = rng.random(n) < 0.2
        e[off] = 0
        e[:, off] = 0
        return e
    e = np.zeros((n, n), np.uint8)
    if kind == "chain":  # the longest path there is, labels in random order
        order = rng.permutation(n)
        e[order[:-1], order[1:]] = 1
    elif kind == "ones":
        e[:] = 1
    return e


@pytest.mark.parametrize("kind", ["sparse", "dense", "idle", "chain", "ones", "empty"])
@pytest.mark.parametrize("n", SIZES)
def test_model(ctx, n, kind):
    e = relation(kind, n)
    want = oracle.tc_model(e)
    bits, st = ctx.tc_closure(e)
    assert np.array_equal(bits, want)
    assert st["model_ones"] == int(np.unpackbits(want.view(np.uint8)).sum())
    assert st["eps_used"] == oracle.tc_eps(e)
    packed, _ = ctx.tc_closure_bits(oracle.pack(e), n)
    assert np.array_equal(packed, want)


@pytest.mark.parametrize("shift", [1, 7, 8, 15])
@pytest.mark.parametrize("n", [33, 250, 1000])
def test_any_alignment_of_device_rows(ctx, n, shift):
    e = relation("sparse", n)
    buf = torch.full((n * n + 32,), 255, dtype=torch.uint8, device="cuda")  # bytes around it are not read as facts
    dev = buf[shift:shift + n * n].view(n, n)
    dev.copy_(torch.from_numpy(e))
    bits, _ = ctx.tc_closure(dev)
    assert np.array_equal(bits.cpu().numpy().view(np.uint64), oracle.tc_model(e))


@pytest.mark.parametrize("n", [5, 130, 700, 1024])
def test_bad_input(ctx, n):
    for i, j in ((0, 0), (n - 1, n - 1), (n // 2, n - 1)):
        e = relation("sparse", n)
        e[i, j] = 2
        with pytest.raises(dl.DLError) as err:
            ctx.tc_closure(e)
        assert err.value.status == dl.DL_EINVAL
    if n % 64:
        packed = oracle.pack(relation("sparse", n)).copy()
        packed[n - 1, -1] |= np.uint64(1) << np.uint64(63)
        with pytest.raises(dl.DLError) as err:
            ctx.tc_closure_bits(packed, n)
        assert err.value.status == dl.DL_EINVAL
    e = relation("sparse", n)
    with pytest.raises(dl.DLError) as err:
        ctx.tc_closure(e, eps=2.0)
    assert err.value.status == dl.DL_EINVAL
    assert np.array_equal(ctx.tc_closure(e)[0], oracle.tc_model(e))


@pytest.mark.parametrize("n", [40, 128, 300, 1000])
def test_bad_input_of_any_row_is_seen(ctx, n):
    """One bad byte (or padding bit) in a row of every warp and CTA, many calls each: the flag is a
    vote of the whole CTA, whichever warp runs first."""
    e = torch.from_numpy(relation("sparse", n)).cuda()
    packed = torch.from_numpy(oracle.pack(relation("sparse", n)).view(np.int64)).cuda()
    for i in range(0, n, max(1, n // 40)):
        for j in (0, n - 1):
            was = int(e[i, j])
            e[i, j] = 2 + i % 250
            for _ in range(3):
                with pytest.raises(dl.DLError) as err:
                    ctx.tc_closure(e)
                assert err.value.status == dl.DL_EINVAL, (i, j)
            e[i, j] = was
        if n % 64 == 0:
            continue  # no padding bits
        was = int(packed[i, -1])
        packed[i, -1] = was | -(1 << 63)
        for _ in range(3):
            with pytest.raises(dl.DLError) as err:
                ctx.tc_closure_bits(packed, n)
            assert err.value.status == dl.DL_EINVAL, i
        packed[i, -1] = was
    want = oracle.tc_model(relation("sparse", n))
    assert np.array_equal(ctx.tc_closure(e)[0].cpu().numpy().view(np.uint64), want)
    assert np.array_equal(ctx.tc_closure_bits(packed, n)[0].cpu().numpy().view(np.uint64), want)


@pytest.mark.parametrize("n", [100, 300, 1000])
def test_refused_calls_leave_host_memory_alone(ctx, n):
    """Bad bytes, padding bits and eps: the caller's output is as it was (an earlier query's model is in
    the workspace)."""
    good = relation("sparse", n)
    ctx.tc_closure(good)
    out = np.full((n, dl.words(n)), 0x5A5A5A5A5A5A5A5A, np.uint64)
    before = out.copy()
    bad = good.copy()
    bad[n // 2, n - 1] = 2
    padded = oracle.pack(good).copy()
    padded[n - 1, -1] |= np.uint64(1) << np.uint64(63)
    for call in (lambda: ctx.tc_closure(bad, out=out), lambda: ctx.tc_closure_bits(padded, n, out=out),
                 lambda: ctx.tc_closure(good, eps=2.0, out=out)):
        with pytest.raises(dl.DLError) as err:
            call()
        assert err.value.status == dl.DL_EINVAL
        assert np.array_equal(out, before)
    ctx.tc_closure(good, out=out)
    assert np.array_equal(out, oracle.tc_model(good))


@pytest.mark.parametrize("kind,n", [("sparse", 300), ("chain", 512), ("chain", 1000)])
def test_packed_host_rows_in_place(ctx, kind, n):
    """The output over the input, also where a long path is handed to the general route."""
    e = relation(kind, n)
    ctx.tc_closure(relation("dense", n))
    rows = oracle.pack(e).copy()
    ctx.tc_closure_bits(rows, n, out=rows)
    assert np.array_equal(rows, oracle.tc_model(e))
