"""Calls of several sizes at once, from serving slots and from contexts on threads of their own: a kernel's
shared-memory limit is shared by all of them and must hold the largest need at any time.  Models equal
the oracle's bits; real solutions are checked by their models."""
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_1608_00139_gb300 import dl, inputs

pytestmark = pytest.mark.gpu


def test_small_closures_of_mixed_sizes_in_slots():
    sizes = [1024, 520, 1000, 600, 1024, 130, 700, 300]
    graphs = [inputs.er_digraph(n, 4.0 / n, n + k) for k, n in enumerate(sizes)]
    want = [oracle.tc_model(e) for e in graphs]
    dev = [torch.from_numpy(e).cuda() for e in graphs]
    with dl.Context(0, max_slots=4) as c:
        for _ in range(12):
            handles = [c.submit(0, d) for d in dev]
            for w, (t, h) in zip(want, handles):
                assert c.poll(t, -1)[0] == dl.DL_OK
                assert np.array_equal(h["bits"].cpu().numpy().view(np.uint64), w)


def run_kind(c, kind, e):
    if kind == "transposed":
        return c.transposed(e, rtilde=True)[0]
    if kind == "sg_real":
        return c.sg_real(e, path="fp64")[1]
    return c.tc_closure(e, path=kind, rtilde=True)[0]


@pytest.mark.parametrize("kind", ["transposed", "mixed", "sg_real"])
def test_contexts_on_threads_of_mixed_sizes(kind):
    def relation(n, seed):  # (with a cycle: same generation takes the series)
        return inputs.er_digraph(n, 1.5 / n if kind == "sg_real" else 4.0 / n, seed)

    def model(e):
        if kind == "transposed":
            return oracle.pack(oracle.trans_model(e).astype(np.uint8))
        return oracle.sg_model(e) if kind == "sg_real" else oracle.tc_model(e)

    work = []
    for sizes in ((1536, 300), (700, 1100), (260, 513)):
        graphs = [relation(n, n) for n in sizes]
        work.append([(torch.from_numpy(e).cuda(), model(e)) for e in graphs])
    errors = []

    def worker(items):
        try:
            with dl.Context(0) as c:
                for _ in range(6):
                    for d, want in items:
                        assert np.array_equal(run_kind(c, kind, d).cpu().numpy().view(np.uint64), want)
        except Exception as err:  # noqa: BLE001
            errors.append(err)

    threads = [threading.Thread(target=worker, args=(items,)) for items in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
