"""Block products whose digit sums and partial sums sit at the limits that the
tensor-core kernel's exactness rests on: 512 terms of a high times a low digit and
a low times a high one share an fp32 accumulator, which holds whole numbers up
to 2^24, and 32768 residues of up to p + p / 64 share a 32-bit word.  The products
are of constants, so the results are known in closed form."""
import numpy as np
import pytest
import torch

from gpu_util import dev2, host



def digits(s):
    """The balanced digits (h, l) of s = 256 h + l with l in [-128, 127]."""
    u = s + 32896
    return (u >> 8) - 128, (u & 255) - 128


def centred(a, p):
    return a - p if a > (p - 1) // 2 else a


def multiply(lib, ctx, p, A, B, prepared):
    m, k = A.shape
    C = torch.full((m, B.shape[1]), -1, dtype=torch.int32, device="cuda")
    Ad = dev2(A, (k + 3) // 4 * 4)
    if prepared:
        prep = lib.BlockPrep(ctx, p, Ad)
        prep.matmul(ctx, dev2(B), C)
        torch.cuda.synchronize()
        prep.close()
    else:
        lib.gfp_matmul_block(ctx, p, Ad, dev2(B), C)
        torch.cuda.synchronize()
    assert lib.gfp_context_check(ctx) == lib.GFP_OK
    return host(C)


def test_digit_pairs_that_reach_the_accumulator_limit():
    """What the cases below drive: 512 terms of 32640 = (128, -128) with itself
    sum to exactly -2^24 in the middle accumulator."""
    assert digits(32640) == (128, -128)
    h, l = digits(32640)
    assert 512 * (h * l + l * h) == -(1 << 24)
    assert digits(-32896) == (-128, -128)


@pytest.mark.gpu
@pytest.mark.parametrize("k", [512, 513, 1024, 4096])
@pytest.mark.parametrize("p", [65521, 65536, 65537, 65789])
def test_middle_sums_at_2_24(lib, ctx, p, k):
    """Rows and columns of constants, so C[i][j] = k a_i b_j: the residues of
    +-32640 and their neighbours, +-(p-1)/2, and (p = 65536, prepared) the one
    whose representative is -32896."""
    vals = [32640, p - 32640, 32639, p - 32639, 32641, p - 32641, (p - 1) // 2, p - (p - 1) // 2, 32512, 128, p - 128,
            1, p - 1, 0]
    a = np.array([vals[i % len(vals)] for i in range(200)], dtype=np.int64)
    b = np.array([vals[(3 * j) % len(vals)] for j in range(64)], dtype=np.int64)
    a[:16] = 32640
    b[:8] = 32640
    want = (k * (a[:, None] * b[None, :] % p)) % p
    A = np.repeat(a[:, None], k, axis=1).astype(np.uint32)
    B = np.repeat(b[None, :], k, axis=0).astype(np.uint32)
    for prepared in (False, True):
        assert np.array_equal(multiply(lib, ctx, p, A, B, prepared), want.astype(np.uint32)), prepared


def drained(p, a, b):
    """The value the kernel's drain adds to a partial sum for 512 terms a b: three
    steps of Horner's rule with a quotient estimated from floor(2^32 / p)."""
    (ha, la), (hb, lb) = digits(centred(a, p)), digits(centred(b, p))
    magic = min((1 << 32) // p, (1 << 31) - 1)
    t = 0
    for s in (512 * ha * hb, 512 * (ha * lb + la * hb), 512 * la * lb):
        t = t * 256 + s
        t -= ((t * magic) >> 32) * p
    return t + p if t < 0 else t


@pytest.mark.gpu
@pytest.mark.parametrize("p", [65521, 65789, 65280])
def test_longest_partial_sums(lib, ctx, p):
    """K = 2^24 terms (the most of one launch, 32768 chunks) of the constants,
    among 4000 pairs, whose chunks add the most to a partial sum."""
    k = 1 << 24
    rng = np.random.default_rng(p)
    pairs = [(int(x), int(y)) for x, y in rng.integers(0, p, size=(4000, 2))]
    a, b = max(pairs, key=lambda q: drained(p, *q))
    assert p - 40 < drained(p, a, b) <= p + p // 64 and drained(p, a, b) * 32768 < 1 << 32
    A, B = np.full((1, k), a, np.uint32), np.full((k, 1), b, np.uint32)
    assert multiply(lib, ctx, p, A, B, False)[0, 0] == k * a * b % p
