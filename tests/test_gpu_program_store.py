"""The matrices that programs keep between their runs: bounded for all programs of a context together, freed
with their program, and given up when any other allocation of the context finds no room."""
import contextlib

import numpy as np
import pytest
import torch

from paper_1608_00139_gb300 import dl

pytestmark = pytest.mark.gpu

TEXT = """r(X,Y) :- e(X,Y).   r(X,Y) :- e(X,Z), r(Z,Y).
          s(X,Y) :- r(X,Y).   s(X,Y) :- s(X,Z), f(Z,Y).
          j(X,Y) :- r(X,Z), s(Z,Y)."""
N = 12000
MATRIX = N * N


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def sparse_relation():
    e = torch.zeros((N, N), dtype=torch.uint8, device="cuda")
    i = torch.arange(0, N - 2, 5, device="cuda")
    e[i, i + 1] = 1
    e[i + 1, i + 2] = 1
    return e


def test_one_bound_for_all_programs():
    e = sparse_relation()
    with dl.Context(0) as c:
        progs, free = [], []
        for _ in range(4):
            p = c.program(TEXT)
            p.set("e", e)
            p.set("f", e)
            p.run()
            progs.append(p)
            free.append(free_bytes())
        # a program's own: two base relations, three models; 2 MiB steps of the allocator
        own = 5 * MATRIX + (64 << 20)
        assert free[2] - free[3] <= own
        assert free[0] - free[3] <= 3 * own + (1 << 30)
        want = progs[0].get("j")
        for p in progs:  # in turn, over matrices that the others' runs pushed out
            p.run()
            assert np.array_equal(p.get("j"), want)
        held = free_bytes()
        for p in progs:
            p.close()
        assert free_bytes() - held >= 4 * 5 * MATRIX + (1 << 30) - 2 * MATRIX


@contextlib.contextmanager
def only(leave):
    """All of the device's free memory taken but `leave` bytes."""
    torch.cuda.empty_cache()
    full = torch.empty(free_bytes() - leave, dtype=torch.uint8, device="cuda")
    yield
    del full
    torch.cuda.empty_cache()


def test_idle_matrices_give_way():
    """A base relation, a workspace and a serving slot's workspace that find no room take that of the
    programs' idle matrices."""
    e = sparse_relation()
    big = torch.zeros((14000, 14000), dtype=torch.uint8, device="cuda")
    big[0, 13999] = 1
    out = torch.empty((14000, dl.words(14000)), dtype=torch.int64, device="cuda")
    with dl.Context(0, max_slots=1, hbm_budget_bytes=16 << 30) as c:
        p = c.program(TEXT)
        p.set("e", e)
        p.set("f", e)
        p.run()
        want = p.get("r")
        small = np.zeros((100, 100), np.uint8)
        t, h = c.submit(0, small)  # (the slot's own set-up)
        assert c.poll(t, -1)[0] == dl.DL_OK
        q = c.program(TEXT)
        with only(200 << 20):  # room for one relation
            q.set("e", e)
            q.set("f", e)
        p.run()
        with only(16 << 20):
            _, st = c.tc_closure(big, out=out)
        assert st["model_ones"] == 1 and int(out[0, 13999 >> 6]) == 1 << (13999 & 63)
        p.run()
        with only(64 << 20):
            t, h = c.submit(0, e)
            assert c.poll(t, -1)[0] == dl.DL_OK
        assert np.array_equal(h["bits"].cpu().numpy().view(np.uint64), want)
        p.run()
        q.run()
        for k in (p, q):
            assert np.array_equal(k.get("r"), want)
