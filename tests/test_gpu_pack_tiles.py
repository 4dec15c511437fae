"""The packing of byte matrices by tiles of rows: sizes around a tile's rows and bytes and the words of
a row, every misalignment of the matrix, bytes around it that are not 0 or 1, and a bad byte at each
place where a piece is cut.  Models equal the oracle's bits (whole numbers: no tolerance)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1608_00139_gb300 import dl, inputs

pytestmark = pytest.mark.gpu

# above 1024 constants (smaller closures pack elsewhere); 4096 and 8192 bytes are tile lines
SIZES = [1025, 1088, 1365, 2047, 2048, 2049, 4095, 4096, 4097, 4111]


def placed(e, off):
    """The matrix `off` bytes into a buffer of 0xFF bytes."""
    n = e.shape[0]
    buf = torch.full((off + n * n + 32,), 0xFF, dtype=torch.uint8, device="cuda")
    view = buf[off:off + n * n].view(n, n)
    view.copy_(torch.from_numpy(e))
    return view


@pytest.mark.parametrize("n", SIZES)
def test_closure_of_misaligned_bytes(ctx, n):
    oracle.set_threads(0)
    off = n % 16 or 3
    e = inputs.er_digraph(n, 1.5 / n, n)
    e[0, 0] = e[n - 1, n - 1] = e[n - 1, 0] = e[0, n - 1] = 1
    ref = oracle.tc_model(e)
    assert np.array_equal(ctx.tc_closure(placed(e, off))[0].cpu().numpy().view(np.uint64), ref)
    assert np.array_equal(ctx.tc_batch([placed(e, 16 - off)])[0][0].cpu().numpy().view(np.uint64), ref)


@pytest.mark.parametrize("n", [1, 3, 17, 100, 1100, 2049])
def test_batch_of_misaligned_bytes(ctx, n):
    oracle.set_threads(0)
    gs = [inputs.er_digraph(n, min(1.0, 1.5 / n), n + k) for k in range(4)]
    outs, _ = ctx.tc_batch([placed(e, 5 * k + 1) for k, e in enumerate(gs)])
    for e, b in zip(gs, outs):
        assert np.array_equal(b.cpu().numpy().view(np.uint64), oracle.tc_model(e))


@pytest.mark.parametrize("n", [1100, 4097])
def test_bad_byte_is_refused(ctx, n):
    e = inputs.er_digraph(n, 1.0 / n, n)
    for i, j in [(0, 0), (0, n - 1), (n - 1, 0), (n - 1, n - 1), (n // 2, 17), (7, n - 1)]:
        d = placed(e, 9)
        for v in (2, 128, 255):
            d[i, j] = v
            for call in (lambda: ctx.tc_closure(d), lambda: ctx.tc_batch([d])):
                with pytest.raises(dl.DLError) as ei:
                    call()
                assert ei.value.status == dl.DL_EINVAL
    assert ctx.tc_closure(placed(e, 9))[1]["model_ones"] >= 0
