"""Block products at the edges of the tensor-core kernel's work split: row
tiles of 128, k-blocks of 64, K ranges of at most eight k-blocks (one range:
results go straight to C), column tiles of 64, rows of A of any alignment, one
context used for several shapes, and K beyond one launch."""
import numpy as np
import pytest
import torch

import gfp_inputs as gi
import oracle
from gpu_util import dev2, host

pytestmark = pytest.mark.gpu


def product(lib, ctx, p, A, B, lda=None, front=0, prepared=False):
    m, k = A.shape
    nb = B.shape[1]
    lda = lda or k
    store = torch.full((front + m * lda,), -1, dtype=torch.int32, device="cuda")
    Ad = store[front:].view(m, lda)[:, :k]
    Ad.copy_(torch.from_numpy(A.view(np.int32)))
    full = torch.full((m + 1, nb + 1), -1, dtype=torch.int32, device="cuda")
    C = full[:m, :nb]
    if prepared:
        prep = lib.BlockPrep(ctx, p, Ad)
        prep.matmul(ctx, dev2(B), C)
        torch.cuda.synchronize()
        prep.close()
    else:
        lib.gfp_matmul_block(ctx, p, Ad, dev2(B), C)
    torch.cuda.synchronize()
    assert lib.gfp_context_check(ctx) == lib.GFP_OK
    out = host(full)
    assert (out[m] == 0xFFFFFFFF).all() and (out[:, nb] == 0xFFFFFFFF).all(), "wrote outside C"
    return out[:m, :nb]


def check(lib, ctx, p, m, k, nb, **kw):
    A = gi.uniform(p, m * k, 92, 0).reshape(m, k)
    B = gi.uniform(p, k * nb, 92, 1).reshape(k, nb)
    assert np.array_equal(product(lib, ctx, p, A, B, **kw), oracle.block(p, A, B)), (p, m, k, nb, kw)


@pytest.mark.parametrize("k", [1, 63, 64, 65, 128, 192, 511, 512, 513, 577, 1024, 1100])
@pytest.mark.parametrize("m,nb", [(1, 1), (127, 63), (128, 64), (129, 65), (300, 130)])
def test_block_split_edges(lib, ctx, m, nb, k):
    for p in (65521, 65789):
        check(lib, ctx, p, m, k, nb)
    check(lib, ctx, 65521, m, k, nb, prepared=True)


@pytest.mark.parametrize("front,pad", [(1, 0), (0, 1), (2, 2), (3, 1), (0, 2)])
def test_block_rows_of_any_alignment(lib, ctx, front, pad):
    """Automatic path: rows that 16-byte loads cannot take go through the same
    kernel with 4-byte loads, directly and through residue passes."""
    for p in (32749, 65521, 2147483647):
        for m, k, nb in ((257, 1030, 64), (130, 514, 33), (700, 2999, 64)):
            check(lib, ctx, p, m, k, nb, lda=k + pad, front=front)


def test_block_many_row_tiles_in_one_range(lib, ctx):
    """More than one row tile per SM against a single K range, and ranges whose
    lengths differ by one k-block."""
    check(lib, ctx, 65521, 152 * 128 + 5, 300, 64)
    check(lib, ctx, 65521, 40 * 128, 64 * 17, 64)
    check(lib, ctx, 4294967291, 6000, 1100, 64)


def test_block_one_context_many_shapes(lib):
    """The context's buffer holds partial sums at its start (zero between
    products) and other operands at its end: shapes that move the border."""
    c = lib.Context(0)
    try:
        for p, m, k, nb in ((65521, 300, 9000, 8), (65521, 5000, 600, 64), (2147483647, 900, 2000, 64),
                            (65521, 9000, 700, 70), (2147483647, 300, 3000, 16), (65521, 9100, 1300, 64)):
            check(lib, c, p, m, k, nb)
    finally:
        c.close()


@pytest.mark.parametrize("p", [65521, 67108859])
def test_block_k_beyond_one_launch(lib, p):
    """K = 2^24 + 65 terms: two launches, the partial sums of the first reduced
    in between (and one modulus after the other for residue passes)."""
    k = (1 << 24) + 65
    A = gi.uniform(p, k, 93, 0).reshape(1, k)
    B = gi.uniform(p, k, 93, 1).reshape(k, 1)
    c = lib.Context(0)
    try:
        c.set_repr(lib.GFP_REPR_F16TC)
        Ad = torch.zeros((1, (k + 3) // 4 * 4), dtype=torch.int32, device="cuda")[:, :k]
        Ad.copy_(torch.from_numpy(A.view(np.int32)))
        C = torch.full((1, 1), -1, dtype=torch.int32, device="cuda")
        lib.gfp_matmul_block(c, p, Ad, dev2(B), C)
        torch.cuda.synchronize()
        assert lib.gfp_context_check(c) == lib.GFP_OK
        assert np.array_equal(host(C), oracle.block(p, A, B))
    finally:
        c.close()


def test_block_graph_replay_after_another_shape(lib):
    """A captured product replays exactly after the context ran products of
    other shapes (their operands never reach the captured one's partial sums)."""
    c = lib.Context(0)
    try:
        p, m, k, nb = 65521, 3000, 1300, 64
        A, B = gi.uniform(p, m * k, 96, 0).reshape(m, k), gi.uniform(p, k * nb, 96, 1).reshape(k, nb)
        want = oracle.block(p, A, B)
        check(lib, c, p, 200, 20000, 64)          # larger tiles of B, smaller result
        Ad, Bd, C = dev2(A), dev2(B), torch.zeros((m, nb), dtype=torch.int32, device="cuda")
        lib.gfp_matmul_block(c, p, Ad, Bd, C)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        s = torch.cuda.Stream()
        with torch.cuda.graph(g, stream=s):
            lib.gfp_matmul_block(c, p, Ad, Bd, C)
        for m2, k2 in ((200, 20000), (64, 15000), (2500, 900)):
            check(lib, c, p, m2, k2, 64)
            C.fill_(-1)
            g.replay()
            torch.cuda.synchronize()
            assert np.array_equal(host(C), want), (m2, k2)
        del g
    finally:
        c.close()
