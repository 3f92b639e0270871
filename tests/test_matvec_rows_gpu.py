"""Matrix-vector products whose rows start at any 4-byte boundary: the kernel
reads the aligned 16-byte vectors inside a row against x kept in planes, adds
the few elements around them by themselves, and keeps two batches of vectors a
lane in flight across rows.  Results equal the oracle bit for bit."""
import numpy as np
import pytest
import torch

import gfp_inputs as gi
import oracle
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


def run(lib, ctx, p, rows, cols, lda, front, repr_=0):
    """A at `front` words past an aligned start, rows lda apart."""
    A = gi.uniform(p, rows * cols, 91, 0).reshape(rows, cols)
    x = gi.uniform(p, cols, 91, 1)
    store = torch.full((front + rows * lda + 1,), -1, dtype=torch.int32, device="cuda")
    view = store[front:front + rows * lda].view(rows, lda)[:, :cols]
    view.copy_(torch.from_numpy(A.view(np.int32)))
    y = torch.full((rows + 1,), -1, dtype=torch.int32, device="cuda")
    ctx.set_repr(repr_)
    try:
        lib.gfp_matvec(ctx, p, view, dev(x), y, lda=lda, rows=rows, cols=cols)
        torch.cuda.synchronize()
    finally:
        ctx.set_repr(0)
    out = host(y)
    assert out[rows] == 0xFFFFFFFF, "wrote past y"
    assert np.array_equal(out[:rows], oracle.matvec(p, A, x)), (p, rows, cols, lda, front, repr_)


# columns at the edges of a vector, of a batch of 32 lanes x 8 vectors, of two
# batches and of the split of a row over warps
@pytest.mark.parametrize("cols", [1, 2, 3, 4, 5, 7, 8, 9, 127, 129, 1023, 1024, 1027, 2049, 8193, 16387, 33001])
@pytest.mark.parametrize("front,pad", [(0, 0), (1, 0), (2, 1), (3, 3), (1, 2)])
def test_matvec_any_row_alignment(lib, ctx, cols, front, pad):
    for p in (65521, 4294967291):
        for rows in (1, 5, 153, 311):
            run(lib, ctx, p, rows, cols, cols + pad, front)


@pytest.mark.parametrize("repr_", [1, 2, 3, 4, 6, 7])
def test_matvec_unaligned_representations(lib, ctx, repr_):
    for cols in (6, 301, 4099):
        run(lib, ctx, 32749, 157, cols, cols + 1, 1, repr_)


def test_matvec_several_windows_of_rows(lib, ctx):
    """More rows per CTA than residues are kept for at a time, and a row wider
    than x fits in shared memory (aligned, and read by 4-byte loads)."""
    run(lib, ctx, 2147483647, 700001, 5, 5, 1)
    run(lib, ctx, 65521, 64, 51300, 51300, 0)
    run(lib, ctx, 65521, 64, 51301, 51301, 3)
