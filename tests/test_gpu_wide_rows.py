"""A closure whose rows' tile and column mask together come just under 48 KB of shared memory, and over it with
the packing kernel's own counts (n around 196 000).  A few short paths, so that the model is known."""
import pytest
import torch

from paper_1608_00139_gb300 import dl

pytestmark = pytest.mark.gpu

N = 196000  # the mask's 3064 words and the tile's 3065: 49 032 bytes of 49 152


def test_tile_and_mask_at_the_limit_of_shared_memory():
    free, _ = torch.cuda.mem_get_info()
    if free < 180 << 30:  # E, two operands' room, three bit matrices: 130 GB
        pytest.skip("needs 180 GB of free device memory")
    path = [3, 100000, 7, N - 1, 64, 131071, 195999 - 64]
    e = torch.zeros((N, N), dtype=torch.uint8, device="cuda")
    for x, y in zip(path[:-1], path[1:]):
        e[x, y] = 1
    try:
        with dl.Context(0) as c:
            bits, st = c.tc_closure(e)
            assert st["model_ones"] == len(path) * (len(path) - 1) // 2
            for k, x in enumerate(path):
                want = torch.zeros(dl.words(N), dtype=torch.int64)
                for y in path[k + 1:]:
                    b = 1 << (y & 63)
                    want[y >> 6] |= b - (1 << 64) if b >> 63 else b
                assert torch.equal(bits[x].cpu(), want), x
            del bits
    finally:
        del e
        torch.cuda.empty_cache()
