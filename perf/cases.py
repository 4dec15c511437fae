"""Performance cases: calls of this library as a program that evaluates Datalog makes them.

A case is a dict of plain values; ``kind`` names the entry point and the rest its sizes and
options.  ``listed()`` holds one case per kind of use, ``draw(rng)`` another one of the same
ranges.  ``prepare`` builds the inputs on the GPU from the seed, ``run`` makes one call through
the public binding and returns everything it computes, ``exact`` gives the real-valued outputs
from plain torch in 64 bits.

One context serves every call of the process, as in a program that answers query after query:
its workspaces stay, the inputs change.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1608_00139_gb300 import dl, inputs

DEV = "cuda"

# Closure, a join, and same generation over the closure: three layers of one program.
PROGRAM = """
    r(X,Y) :- e(X,Y).   r(X,Y) :- e(X,Z), r(Z,Y).
    sg(X,Y) :- r(X,Y).  sg(X,Y) :- p(X,Z), sg(Z,W), p(Y,W).
    j(X,Y) :- r(X,Z), sg(Z,Y).
"""


def listed():
    return [
        # an interactive query on a small relation: latency and launches are all there is
        {"name": "closure_256", "kind": "closure", "graph": "er", "n": 256, "degree": 5.12, "idle": 0.0,
         "packed": False},
        # the size of the paper's tables (N = 1000), a ragged one, with the relation kept bit-packed;
        # some constants of the domain belong to other relations only
        {"name": "closure_packed_1000", "kind": "closure", "graph": "er", "n": 1000, "degree": 10.0, "idle": 0.02,
         "packed": True},
        # the ordinary closure: an Erdos-Renyi digraph with a giant component (p = 1e-3)
        {"name": "closure_8192", "kind": "closure", "graph": "er", "n": 8192, "degree": 8.192, "idle": 0.0,
         "packed": False},
        # the largest request of the serving stream: a citation-like graph with hubs
        {"name": "closure_pa_16384", "kind": "closure", "graph": "pa", "n": 16384, "degree": 5.0, "idle": 0.0,
         "packed": False},
        # a whole program: three layers over two base relations
        {"name": "program_2048", "kind": "program", "n": 2048, "degree": 1.0},
        # the real solution on the tensor cores, dense relation (p = 1e-2)
        {"name": "mixed_dense_8192", "kind": "mixed", "n": 8192, "degree": 81.92},
        # the tail recursive class with its real solution: a general right-hand side, sparse relations
        {"name": "tail_mixed_8192", "kind": "tail", "n": 8192, "degree": 8.192, "degree_a": 0.8192},
        # the real solution in plain FP64 at the size of the paper's tables
        {"name": "fp64_1000", "kind": "fp64", "n": 1000, "degree": 10.0},
        # same generation on a forest with a few extra edges
        {"name": "sg_4096", "kind": "sg", "graph": "forest", "n": 4096},
        # ... and its real solution with the model
        {"name": "sg_real_4096", "kind": "sg_real", "n": 4096},
        # the transposed class with its real solution
        {"name": "transposed_4096", "kind": "transposed", "n": 4096, "degree": 4.096},
        # many closures of uneven size in one call
        {"name": "batch_1024", "kind": "batch", "count": 1024, "n_hi": 2048, "sizes_seed": 1000},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["closure", "closure", "closure", "program", "mixed", "tail", "fp64", "sg", "sg_real",
                       "transposed", "batch"])
    deg = lambda lo, hi: round(_log(rng, lo, hi), 3)  # noqa: E731
    if kind == "closure":
        return {"kind": kind, "graph": rng.choice(["er", "er", "pa"]), "n": int(_log(rng, 200, 16384)),
                "degree": deg(0.8, 82.0), "idle": 0.02, "packed": rng.random() < 0.3}
    if kind == "program":
        return {"kind": kind, "n": int(_log(rng, 256, 3000)), "degree": deg(0.5, 4.0)}
    if kind == "mixed":
        return {"kind": kind, "n": int(_log(rng, 1000, 8192)), "degree": deg(0.8, 82.0)}
    if kind == "tail":
        return {"kind": kind, "n": int(_log(rng, 1000, 8192)), "degree": deg(0.8, 20.0), "degree_a": deg(0.5, 8.0)}
    if kind == "fp64":
        return {"kind": kind, "n": int(_log(rng, 300, 1500)), "degree": deg(0.8, 82.0)}
    if kind == "sg":
        return {"kind": kind, "graph": rng.choice(["forest", "forest", "pa"]), "n": int(_log(rng, 512, 8192))}
    if kind == "sg_real":
        return {"kind": kind, "n": int(_log(rng, 512, 4096))}
    if kind == "transposed":
        return {"kind": kind, "n": int(_log(rng, 512, 4096)), "degree": deg(1.0, 8.0)}
    return {"kind": kind, "count": int(_log(rng, 64, 1024)), "n_hi": rng.randrange(512, 2049),
            "sizes_seed": rng.randrange(1, 100000)}


_CTX = None


def _context():
    """The context that such a program opens once and keeps."""
    global _CTX
    if _CTX is None:
        _CTX = dl.Context(0)
    return _CTX


def _generator(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _er(n, degree, g, idle=0.0):
    """Erdos-Renyi digraph of mean out-degree ``degree``, no self-loops, as 0/1 bytes; a share
    ``idle`` of the constants has no facts."""
    p = min(1.0, degree / max(n, 1))
    e = torch.empty((n, n), dtype=torch.uint8, device=DEV)
    for r in range(0, n, 2048):
        e[r:r + 2048] = torch.rand((min(2048, n - r), n), generator=g, device=DEV) < p
    e.fill_diagonal_(0)
    if idle > 0.0:
        off = torch.rand(n, generator=g, device=DEV) < idle
        e[off] = 0
        e[:, off] = 0
    return e


def _pa(n, seed):
    """Preferential-attachment DAG with Zipf out-degrees (hubs), the stand-in for real networks."""
    return torch.from_numpy(inputs.pa_dag_into(np.zeros((n, n), np.uint8), seed)).to(DEV)


def _forest(n, seed):
    return torch.from_numpy(inputs.forest_dag(n, seed)).to(DEV)


def _pack(e):
    """n x ceil(n/64) int64 words, least significant bit first."""
    n = e.shape[0]
    w = dl.words(n)
    out = torch.empty((n, w), dtype=torch.int64, device=DEV)
    shifts = torch.arange(64, device=DEV, dtype=torch.int64)
    for r in range(0, n, 1024):
        rows = torch.nn.functional.pad(e[r:r + 1024], (0, 64 * w - n)).view(-1, w, 64).to(torch.int64)
        out[r:r + 1024] = (rows << shifts).sum(dim=2)
    return out


def prepare(case, seed):
    kind, n = case["kind"], case.get("n")
    s = {"kind": kind, "ctx": _context(), "n": n}
    if kind == "closure":
        e = _pa(n, seed) if case["graph"] == "pa" else _er(n, case["degree"], _generator(seed, 1), case["idle"])
        s["packed"] = case["packed"]
        s["e"] = _pack(e) if case["packed"] else e
    elif kind in ("mixed", "fp64", "transposed"):
        s["e"] = _er(n, case["degree"], _generator(seed, 1))
    elif kind == "tail":
        s["e"] = _er(n, case["degree"], _generator(seed, 1))
        s["a"] = _er(n, case["degree_a"], _generator(seed, 2))
    elif kind in ("sg", "sg_real"):
        s["p"] = _pa(n, seed) if case.get("graph") == "pa" else _forest(n, seed)
    elif kind == "program":
        s["program"] = s["ctx"].program(PROGRAM)
        s["program"].set("e", _er(n, case["degree"], _generator(seed, 1)))
        s["program"].set("p", _forest(n, seed))
    else:  # batch: all instances back to back in one buffer
        specs = inputs.batch_specs(case["count"], case["sizes_seed"], n_hi=case["n_hi"])
        ns = np.array([k for k, _, _ in specs], dtype=np.int32)
        size = (ns.astype(np.int64) ** 2 + 255) // 256 * 256
        off = np.concatenate(([0], np.cumsum(size)[:-1]))
        s["buf"] = torch.zeros(int(size.sum()), dtype=torch.uint8, device=DEV)
        g = _generator(seed, 1)
        for (k, p, _), o in zip(specs, off.tolist()):
            m = s["buf"][o:o + k * k].view(k, k)
            torch.lt(torch.rand((k, k), generator=g, device=DEV), p, out=m)
            m.fill_diagonal_(0)
        s["ns"], s["off"] = ns, off.astype(np.uint64)
    return s


def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind == "closure":
        if state["packed"]:
            return {"bits": ctx.tc_closure_bits(state["e"], state["n"])[0]}
        return {"bits": ctx.tc_closure(state["e"])[0]}
    if kind in ("mixed", "fp64"):
        bits, _, x = ctx.tc_closure(state["e"], path=kind, rtilde=True)
        return {"bits": bits, "x": x}
    if kind == "tail":
        bits, _, x = ctx.tail_recursive(state["e"], state["a"], path="mixed", rtilde=True)
        return {"bits": bits, "x": x}
    if kind == "sg":
        return {"bits": ctx.sg_least_model(state["p"])[0]}
    if kind == "sg_real":
        x, bits, _ = ctx.sg_real(state["p"])
        return {"bits": bits, "x": x}
    if kind == "transposed":
        bits, _, x = ctx.transposed(state["e"], rtilde=True)
        return {"bits": bits, "x": x}
    if kind == "program":
        prog = state["program"]
        prog.run()
        return {p: prog.get(p, device=True) for p in ("r", "sg", "j")}
    return {"bits": ctx.tc_batch_flat(state["buf"], state["ns"], state["off"])[0]}


def work(case):
    """Inputs read once, outputs written once; for the real solutions of the closure form the flops
    of the dense direct solve (8/3 n^3), for the two-sided and transposed ones those of one
    application of their operator."""
    kind = case["kind"]
    if kind == "batch":
        ns = [k for k, _, _ in inputs.batch_specs(case["count"], case["sizes_seed"], n_hi=case["n_hi"])]
        return {"bytes": float(sum(k * k + 8 * k * dl.words(k) for k in ns)), "flops": 0.0}
    n = case["n"]
    nn, bits = float(n) * n, 8.0 * n * dl.words(n)
    if kind == "closure":
        return {"bytes": (bits if case["packed"] else nn) + bits, "flops": 0.0}
    if kind == "program":
        return {"bytes": 2 * nn + 3 * bits, "flops": 0.0}
    if kind == "sg":
        return {"bytes": nn + bits, "flops": 0.0}
    if kind == "sg_real":
        return {"bytes": 9 * nn + bits, "flops": 2 * nn}
    if kind == "transposed":
        return {"bytes": 9 * nn + bits, "flops": 2 * nn * case["degree"]}
    return {"bytes": (2 if kind == "tail" else 1) * nn + 8 * nn + bits, "flops": 8.0 / 3.0 * nn * n}


def _series(step, n):
    """The increasing series X <- step(X) from 0, until a step changes nothing any more."""
    x = torch.zeros((n, n), dtype=torch.float64, device=DEV)
    for _ in range(2000):
        y = step(x)
        if float((y - x).abs().max()) <= 1e-19:
            return y
        x = y
    return None


def exact(case, seed):
    """The real-valued outputs (Proposition 1 and its analogues) in FP64 by plain torch."""
    kind = case["kind"]
    if kind in ("closure", "sg", "program", "batch"):
        return None  # bits: whole numbers
    s = prepare(case, seed)
    n = case["n"]
    if kind in ("mixed", "fp64", "tail"):
        e = s["e"].double()
        eps = 1.0 / (1.0 + float(e.sum(dim=1).max()))
        rhs = eps * (s["a"].double() if kind == "tail" else e)
        a = torch.eye(n, dtype=torch.float64, device=DEV) - eps * e
        return {"bits": None, "x": torch.linalg.solve(a, rhs)}
    m = (s["p"] if kind == "sg_real" else s["e"]).double()
    d = float(m.sum(dim=1).max())
    sp = m.to_sparse_csr()
    if kind == "sg_real":  # S = eps (I + P S P^T)
        eps = 1.0 / (1.0 + d * d)
        eye = torch.eye(n, dtype=torch.float64, device=DEV)
        x = _series(lambda x: eps * (eye + sp @ (sp @ x.t().contiguous()).t().contiguous()), n)
    else:  # R = eps (R1 + R1 R^T)
        eps = 1.0 / (1.0 + d)
        x = _series(lambda x: eps * (m + sp @ x.t().contiguous()), n)
    return None if x is None else {"bits": None, "x": x}
