"""Block products back to back on one stream, each reading what the one before
it wrote: as A, as B, and through two buffers by turns, so that memory a kernel has
read is written and read again a few launches later."""
import re

import numpy as np
import pytest
import torch

import gfp_inputs as gi
import oracle
from gpu_util import dev2, host
from test_block_registers_cpu import source


def test_product_kernel_waits_before_it_reads():
    """The kernel is placed while the one before it runs, whose writes and whose
    predecessors' it may only read behind griddepcontrol.wait: each role that
    touches global memory starts with it (no GPU needed)."""
    src = source()
    kernel = src[src.index("k_block_tc(const __grid_constant__ Args a)"):src.index("struct PrepB")]
    cuts = [kernel.index(c) for c in ("if (warp < W_EPI0) {", "} else if (warp == W_MMA) {", "} else if (warp > W_MMA) {")]
    cuts.append(kernel.index("} else {\n", kernel.index("bulk_g2s(")))
    conv, mma, bprod, epi = (kernel[i:j] for i, j in zip(cuts, cuts[1:] + [None]))
    reads = {"conv": (conv, "ld.load("), "bprod": (bprod, "bulk_g2s("), "epi": (epi, "dst")}
    for name, (text, first) in reads.items():
        assert "griddepcontrol.wait" in text and text.index("griddepcontrol.wait") < text.index(first), name
    assert not re.search(r"ld\.load|bulk_g2s|Cacc|a\.A\b|a\.C\b", mma)


@pytest.mark.gpu
@pytest.mark.parametrize("lda_pad", [0, 1])
@pytest.mark.parametrize("side", ["A", "B"])
@pytest.mark.parametrize("p,n", [(65521, 256), (65521, 640), (65789, 640), (2147483647, 640)])
def test_products_of_products(lib, ctx, p, n, side, lda_pad):
    steps = 8
    X = gi.uniform(p, n * n, 97, 0).reshape(n, n)
    M = gi.uniform(p, n * n, 97, 1).reshape(n, n)
    want = [X]
    for _ in range(steps):
        want.append(oracle.block(p, want[-1], M) if side == "A" else oracle.block(p, M, want[-1]))
    Md = dev2(M, n + lda_pad)
    bufs = [torch.zeros((n, n + lda_pad), dtype=torch.int32, device="cuda")[:, :n] for _ in range(2)]
    x0 = dev2(X)
    lib.gfp_matmul_block(ctx, p, *((x0, Md) if side == "A" else (Md, x0)), bufs[0])   # the workspace grows here
    for again in range(5):
        bufs[0].copy_(x0)
        for t in range(steps):
            src, dst = bufs[t & 1], bufs[1 - (t & 1)]
            lib.gfp_matmul_block(ctx, p, *((src, Md) if side == "A" else (Md, src)), dst)
        torch.cuda.synchronize()
        assert np.array_equal(host(bufs[steps & 1]), want[steps]), again
        assert np.array_equal(host(bufs[(steps - 1) & 1]), want[steps - 1]), again
    assert lib.gfp_context_check(ctx) == lib.GFP_OK
