"""The mixed path with R~ where device memory is short of the kept sums (8 np^2 bytes): every residual is then
formed as a whole, and later buffers of the call may take the sums' room.  The solution is held to the
equation as in test_gpu_mixed_updates."""
import pytest
import torch

from paper_1608_00139_gb300 import dl, inputs
from tests.test_gpu_mixed_updates import check

pytestmark = pytest.mark.gpu

N, NP = 3000, 3072


def solve(c, e, a):
    if a is None:
        return c.tc_closure(e, path="mixed", rtilde=True)
    return c.tail_recursive(e, a, path="mixed", rtilde=True)


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


# gathered sums, sums as products, bands; a right-hand side of its own or not
@pytest.mark.parametrize("degree", [4.0, 31.0, 90.0])
@pytest.mark.parametrize("tail", [False, True])
def test_short_of_the_sums(degree, tail):
    e = inputs.er_digraph(N, degree / N, int(degree))
    a = inputs.er_digraph(N, 3.0 / N, 5) if tail else None
    dev = torch.from_numpy(e).cuda()
    deva = torch.from_numpy(a).cuda() if tail else None
    with dl.Context(0) as warm:  # (loads the kernels)
        solve(warm, dev, deva)
    torch.cuda.empty_cache()
    with dl.Context(0) as c:
        before = free_bytes()
        want, _, x0 = solve(c, dev, deva)
        used = before - free_bytes() - x0.numel() * 8
    check(e, x0, a)
    out = torch.empty((N, N), dtype=torch.float64, device="cuda"), torch.empty_like(want)  # room for the next results
    del out, x0
    short = 8 * NP * NP * 3 // 4
    filler = torch.empty(free_bytes() - (used - short), dtype=torch.uint8, device="cuda")
    try:
        with dl.Context(0) as c:
            bits, _, x = solve(c, dev, deva)
            assert torch.equal(bits, want)
            again, _, _ = solve(c, dev, deva)
            assert torch.equal(again, want)
    finally:
        del filler
        torch.cuda.empty_cache()
    check(e, x, a)
