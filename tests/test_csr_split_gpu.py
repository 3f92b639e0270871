"""Sparse-row block products with few rows: two, four or eight warps share a row
(each a run of its nonzeros in steps of eight) and meet in shared memory.  Row
counts at the limits of each split, rows with fewer nonzeros than warps, empty
rows, rows at the edges of a chunk of 32, several 64-column groups."""
import numpy as np
import pytest
import torch

import gfp_inputs as gi
import oracle
from gpu_util import dev, dev2, host

pytestmark = pytest.mark.gpu


def run(lib, ctx, p, k, nb, lengths, repr_=0):
    rng = np.random.default_rng(95)
    cols = [np.sort(rng.choice(k, size=n, replace=False)).astype(np.uint32) for n in lengths]
    row_ptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.uint32)
    col = np.concatenate(cols + [np.zeros(1, np.uint32)])
    val = rng.integers(0, p, size=col.size, dtype=np.uint64).astype(np.uint32)
    B = gi.uniform(p, k * nb, 95, 1).reshape(k, nb)
    C = torch.full((len(lengths) + 1, nb), -1, dtype=torch.int32, device="cuda")
    ctx.set_repr(repr_)
    try:
        lib.gfp_matmul_block_csr(ctx, p, k, dev(row_ptr), dev(col), dev(val), dev2(B), C[:len(lengths)])
        torch.cuda.synchronize()
    finally:
        ctx.set_repr(0)
    out = host(C)
    assert (out[len(lengths)] == 0xFFFFFFFF).all(), "wrote past C"
    n = int(row_ptr[-1])
    assert np.array_equal(out[:-1], oracle.csr(p, row_ptr, col[:n], val[:n], B)), (p, k, nb, len(lengths), repr_)


EDGES = [0, 1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 100, 127, 128, 129, 255, 257, 400]


@pytest.mark.parametrize("rows", [1, 2, 3, 17, 607, 608, 609, 1216, 1217, 2432, 2433])
def test_split_row_counts(lib, ctx, rows):
    for p in (65521, 4294967291):
        run(lib, ctx, p, 500, 64, [EDGES[i % len(EDGES)] for i in range(rows)])


@pytest.mark.parametrize("repr_", [0, 1, 2, 3, 6, 7])
@pytest.mark.parametrize("nb", [4, 64, 68, 132])
def test_split_columns_and_representations(lib, ctx, repr_, nb):
    run(lib, ctx, 2147483647, 700, nb, EDGES[::-1] + [699, 0, 512], repr_)
