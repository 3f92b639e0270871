"""Matrix-vector products at the edges between the forms of the kernel: rows read
word by word, short rows in twice the warps, splits of a row over numbers of warps
that do not divide a CTA's (some warps then have no row), and rows whose x does not
fit shared memory; the projection fused into each."""
import numpy as np
import pytest
import torch

import gfp_inputs as gi
import oracle
from gpu_util import dev, dev2, host
from test_matvec_rows_gpu import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [60, 63, 64, 65, 68, 255, 256, 257, 260])
@pytest.mark.parametrize("front,pad", [(0, 0), (1, 1), (2, 2)])
def test_short_rows(lib, ctx, cols, front, pad):
    for p in (65521, 2147483647):
        for rows in (1, 33, 153, 5000, 20011):
            run(lib, ctx, p, rows, cols, cols + pad, front)


# just above what one batch of 1, 2, 4, 5, ... warps takes: splits over 2, 3, 5, 8
# and 16 warps
@pytest.mark.parametrize("cols", [1028, 2100, 4100, 4500, 5124, 6148, 7172, 8196, 9220, 12292, 16380])
@pytest.mark.parametrize("front,pad", [(0, 0), (3, 1)])
def test_rows_over_any_number_of_warps(lib, ctx, cols, front, pad):
    for p in (65521, 4294967291):
        for rows in (1, 152 * 3, 2500):
            run(lib, ctx, p, rows, cols, cols + pad, front)


@pytest.mark.parametrize("cols", [51197, 51200, 51201, 51204, 60000])
@pytest.mark.parametrize("front,pad", [(0, 0), (0, 1), (3, 0)])
def test_rows_beyond_shared_memory(lib, ctx, cols, front, pad):
    for p in (65521, 2147483647):
        for rows in (1, 70, 331):
            run(lib, ctx, p, rows, cols, cols + pad, front)


@pytest.mark.parametrize("repr_", [1, 2, 3, 4, 6, 7])
def test_forms_in_each_representation(lib, ctx, repr_):
    for cols in (13, 64, 200, 4500, 51300):
        for pad in (0, 1):
            run(lib, ctx, 32749, 157, cols, cols + (-cols) % 4 + pad, 0, repr_)


@pytest.mark.parametrize("n", [5, 64, 200, 257, 1100, 4500])
@pytest.mark.parametrize("pad", [0, 1])
def test_projection_in_each_form(lib, ctx, n, pad):
    p, iters = 2147483647, 3
    A = gi.uniform(p, n * n, 94, 0).reshape(n, n)
    x, u = gi.uniform(p, n, 94, 1), gi.uniform(p, n, 94, 2)
    want, v = [], x
    for _ in range(iters + 1):
        want.append(oracle.dot(p, u, v))
        v = oracle.matvec(p, A, v)
    seq = torch.full((iters + 1,), -1, dtype=torch.int32, device="cuda")
    Ad = dev2(A, n + (-n) % 4 + pad)
    for _ in range(2):
        lib.gfp_matvec_sequence(ctx, p, Ad, dev(x), dev(u), seq, iters)
        torch.cuda.synchronize()
        assert host(seq).tolist() == [int(w) for w in want]
