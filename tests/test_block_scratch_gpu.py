"""Block products by the scratch they have: B's tiles for one residue modulus at a
time where those of all would be too large; and calls that need nothing of the
context, on several streams at once and captured without a call before."""
import threading

import numpy as np
import pytest
import torch

import gfp_inputs as gi
import oracle
from gpu_util import dev2, host

pytestmark = pytest.mark.gpu


def test_tiles_of_b_for_one_modulus_at_a_time(lib):
    """20 x 4096 by 4096 x 16448 over GF(2^31 - 1): 1.3 GiB of tiles for the five
    moduli.  Checked in the columns at the edges and some between."""
    p, m, k, nb = 2147483647, 20, 4096, 16448
    A = gi.uniform(p, m * k, 98, 0).reshape(m, k)
    B = gi.uniform(p, k * nb, 98, 1).reshape(k, nb)
    cols = np.r_[0:70, 8000:8070, nb - 70:nb]
    c = lib.Context(0)
    try:
        C = torch.full((m, nb), -1, dtype=torch.int32, device="cuda")
        Bd = dev2(B)
        for _ in range(2):
            n0 = lib.gfp_launch_count(c)
            lib.gfp_matmul_block(c, p, dev2(A), Bd, C)
            torch.cuda.synchronize()
            assert lib.gfp_launch_count(c) - n0 == 3 * 5 + 1
            assert lib.gfp_context_check(c) == lib.GFP_OK
            assert np.array_equal(host(C)[:, cols], oracle.block(p, A, np.ascontiguousarray(B[:, cols])))
    finally:
        c.close()


# rows of A that 16-byte loads cannot take, and a small product over a large modulus
FREE = [(65521, 700, 2999, 64), (65789, 3001, 5003, 40), (2147483647, 513, 1031, 64), (2147483647, 1024, 1024, 64),
        (65521, 129, 301, 33)]


def operands(p, m, k, nb, n):
    A = [gi.uniform(p, m * k, 99 + i, 0).reshape(m, k) for i in range(n)]
    B = [gi.uniform(p, k * nb, 99 + i, 1).reshape(k, nb) for i in range(n)]
    want = [oracle.block(p, a, b) for a, b in zip(A, B)]
    C = [torch.full((m, nb), -1, dtype=torch.int32, device="cuda") for _ in range(n)]
    return [dev2(a) for a in A], [dev2(b) for b in B], C, want


@pytest.mark.parametrize("p,m,k,nb", FREE)
def test_streams_of_one_context_at_once(lib, p, m, k, nb):
    """The same context on three streams, nothing ordering them, several products on
    each behind one another; one more stream runs products through the context's
    buffer."""
    n = 3
    A, B, C, want = operands(p, m, k, nb, n)
    A4, B4, C4, want4 = operands(65521, 1000, 2000, 64, 1)
    c = lib.Context(0)
    try:
        streams = [torch.cuda.Stream() for _ in range(n + 1)]
        torch.cuda.synchronize()
        for _ in range(4):
            for x in C + C4:
                x.fill_(-1)
            torch.cuda.synchronize()
            for _ in range(6):
                for i in range(n):
                    lib.gfp_matmul_block(c, p, A[i], B[i], C[i], stream=streams[i])
                lib.gfp_matmul_block(c, 65521, A4[0], B4[0], C4[0], stream=streams[n])
            torch.cuda.synchronize()
            for i in range(n):
                assert np.array_equal(host(C[i]), want[i]), i
            assert np.array_equal(host(C4[0]), want4[0])
        assert lib.gfp_context_check(c) == lib.GFP_OK
    finally:
        c.close()


@pytest.mark.parametrize("p,m,k,nb", FREE[:4])
def test_threads_of_one_context_at_once(lib, p, m, k, nb):
    """Two threads with a stream each and no order between them, and two on one
    stream."""
    for streams in ([torch.cuda.Stream(), torch.cuda.Stream()], [torch.cuda.Stream()] * 2):
        A, B, C, want = operands(p, m, k, nb, 2)
        c = lib.Context(0)
        try:
            torch.cuda.synchronize()
            errors = []

            def work(i):
                try:
                    for _ in range(20):
                        lib.gfp_matmul_block(c, p, A[i], B[i], C[i], stream=streams[i])
                except Exception as e:
                    errors.append(e)

            threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
            torch.cuda.synchronize()
            assert not errors
            assert all(np.array_equal(host(C[i]), want[i]) for i in range(2))
            assert lib.gfp_context_check(c) == lib.GFP_OK
        finally:
            c.close()


@pytest.mark.parametrize("p,m,k,nb", FREE)
def test_captured_without_a_call_before(lib, p, m, k, nb):
    A, B, C, want = operands(p, m, k, nb, 2)
    c = lib.Context(0)
    try:
        g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(g, stream=s):
            lib.gfp_matmul_block(c, p, A[0], B[0], C[0])
        C[0].fill_(-1)
        other = torch.cuda.Stream()
        torch.cuda.synchronize()
        for _ in range(3):      # replays beside calls of the same context
            g.replay()
            for _ in range(3):
                lib.gfp_matmul_block(c, p, A[1], B[1], C[1], stream=other)
        torch.cuda.synchronize()
        assert np.array_equal(host(C[0]), want[0]) and np.array_equal(host(C[1]), want[1])
        del g
    finally:
        c.close()


@pytest.mark.parametrize("p,m,k,nb", FREE[:3])
def test_beside_a_capture(lib, p, m, k, nb):
    """While another stream is being captured (in the mode that watches all
    threads), such a call runs on a stream of its own, the first of a context too."""
    A, B, C, want = operands(p, m, k, nb, 1)
    c, c2 = lib.Context(0), lib.Context(0)
    try:
        g, s, other = torch.cuda.CUDAGraph(), torch.cuda.Stream(), torch.cuda.Stream()
        x = torch.zeros(1000, dtype=torch.int32, device="cuda")
        lib.gfp_matmul_block(c2, p, A[0], B[0], C[0])     # kernels loaded
        C[0].fill_(-1)
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=s, capture_error_mode="global"):
            x.add_(1)
            lib.gfp_matmul_block(c, p, A[0], B[0], C[0], stream=other)
            x.add_(1)
        torch.cuda.synchronize()
        assert np.array_equal(host(C[0]), want[0])
        g.replay()
        torch.cuda.synchronize()
        assert int(x[0]) == 2
        del g
    finally:
        c.close()
        c2.close()
