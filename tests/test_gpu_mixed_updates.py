"""The mixed path's residual updates: R~ on both sides of the lines between gathered and product
updates and at the sums' largest sizes, against the equation itself in FP64 on the host or device
(A X = eps E, A X = eps A1).  Tolerance: the solver's own stopping rule max|R| <= 1e-13 eps, plus
the FP64 evaluation of the equation here, (row length + 2) units of 2^-53 of eps max|X| at most."""
import numpy as np
import pytest
import torch

from paper_1608_00139_gb300 import inputs

pytestmark = pytest.mark.gpu


def check(e, x, rhs=None):
    ed = torch.from_numpy(e).cuda().double()
    x = torch.as_tensor(x).cuda().double()
    eps = 1.0 / (1.0 + float(ed.sum(dim=1).max()))
    b = ed if rhs is None else torch.from_numpy(rhs).cuda().double()
    r = eps * (b + ed @ x) - x
    top = float(ed.sum(dim=1).max()) + 2
    bound = 1e-13 * eps + (top + 2) * 2.0 ** -53 * eps * top * max(float(x.abs().max()), 1.0)
    assert float(r.abs().max()) <= bound


def hub(n, degree, seed):
    """A sparse graph with one constant that reaches all others."""
    e = inputs.er_digraph(n, degree / n, seed)
    e[n // 3, :] = 1
    return e


@pytest.mark.parametrize("e", [
    inputs.er_digraph(300, 0.02, 1), inputs.er_digraph(257, 0.5, 2), np.ones((200, 200), np.uint8),
    inputs.er_digraph(1000, 0.0088, 3), inputs.er_digraph(1000, 0.0095, 4), inputs.er_digraph(1500, 0.4, 5),
    inputs.er_digraph(2049, 0.002, 6), inputs.er_digraph(2049, 0.05, 7), hub(1100, 1.5, 8), hub(1100, 20.0, 9),
    np.zeros((70, 70), np.uint8)], ids=lambda e: f"{e.shape[0]}_{int(e.sum())}")
def test_mixed_solution_solves_the_equation(ctx, e):
    d = torch.from_numpy(e).cuda()
    _, _, x = ctx.tc_closure(d, path="mixed", rtilde=True)
    check(e, x)
    a = inputs.er_digraph(e.shape[0], 0.01, 99)
    _, _, x = ctx.tail_recursive(d, torch.from_numpy(a).cuda(), path="mixed", rtilde=True)
    check(e, x, a)


@pytest.mark.parametrize("n,p", [(9000, 0.5), (8500, 0.0005)])
def test_mixed_rows_of_more_than_8192_ones(ctx, n, p):
    """The product's slices are cut shorter where a row has more than 8191 ones."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    d = (torch.rand((n, n), generator=g, device="cuda") < p).to(torch.uint8)
    d[7, :] = 1
    _, _, x = ctx.tc_closure(d, path="mixed", rtilde=True)
    check(d.cpu().numpy(), x)
