"""Device memory of the block products' host code, against a stand-in for the CUDA
runtime (no GPU needed): what is asked for, and what a failed allocation leaves."""
import fake_cuda


def test_smaller_buffer_after_a_failed_allocation(lib):
    """A context's buffer is asked for at the size of its largest parts; where that
    does not fit, this product's parts alone do, and the product runs to its end."""
    for p, last in ((65521, "k_block_finish"), (2147483647, "k_block_crt")):
        fake_cuda.run(f"""
c = context()
assert L.gfp_set_repr(c, g.GFP_REPR_F16TC) == 0             # the context's buffer for all of them
assert block(c, {p}, 64, 4194304, 64) == 0                  # large tiles of B
assert F.fake_used() > 1 << 30
F.fake_room(F.fake_used() + (900 << 20))
F.fake_events()
assert block(c, {p}, 1 << 22, 1024, 8) == 0                 # large workspace: the two together do not fit
ks = kernels()
assert ks[-1].startswith("{last}"), ks
assert block(c, {p}, 256, 256, 64) == 0
""")


def test_failed_allocation_is_not_reported_by_the_next_call(lib):
    fake_cuda.run("""
c = context()
F.fake_room(F.fake_used() + (1 << 20))
out = ctypes.c_void_p()
for _ in range(2):
    assert L.gfp_set_repr(c, g.GFP_REPR_F16TC) == 0
    assert block(c, 65521, 1 << 20, 512, 64) == g.GFP_ERR_NOMEM
    assert L.gfp_set_repr(c, 0) == 0
    assert L.gfp_dot(c, 65521, 1024, A, B, C, 0) == 0
    assert L.gfp_block_prepare(c, 65521, 1 << 20, 512, A, 512, ctypes.byref(out)) == g.GFP_ERR_NOMEM
    assert L.gfp_dot(c, 65521, 1024, A, B, C, 0) == 0
    assert L.gfp_matvec(c, 65521, 1024, 1024, A, 1024, B, C, 0) == 0
""")


def test_tiles_of_b_for_one_modulus_where_all_would_be_too_large(lib):
    """The digit tiles of B take 4 bytes an entry and modulus: those of all moduli
    are made at once up to 1 GiB, and one modulus at a time above that or where
    there is no room."""
    fake_cuda.run("""
p = 2147483647
c = context()
base = F.fake_used()
# small: one launch for all moduli
assert block(c, p, 512, 8192, 64) == 0
ks = kernels()
passes = count(ks, "k_block_tc")
assert passes >= 5 and count(ks, "k_block_prep_b") == 1 and count(ks, "k_block_crt") == 1
# 16384 x 8192: 512 MiB a modulus
assert block(c, p, 512, 16384, 8192) == 0
ks = kernels()
assert count(ks, "k_block_tc") == count(ks, "k_block_prep_b") == passes, ks
tiles, sums = 4 * 16384 * 8192, 4 * 512 * 8192
assert F.fake_used() - base < 1.01 * (tiles + (passes + 1) * sums)
# no room for the tiles of all: the product still runs
assert L.gfp_context_destroy(c) == 0
c = context()
tiles, sums = 4 * 16384 * 1024, 4 * 512 * 1024
F.fake_room(F.fake_used() + int(1.01 * (tiles + (passes + 1) * sums)))
F.fake_events()
assert block(c, p, 512, 16384, 1024) == 0
ks = kernels()
assert count(ks, "k_block_tc") == count(ks, "k_block_prep_b") == passes and ks[-1].startswith("k_block_crt"), ks
# under capture the tiles that fit are used, nothing is allocated
F.fake_room(1 << 40)
F.fake_capture(1)
assert block(c, p, 512, 16384, 1024, stream=CAPTURING) == 0
assert count(kernels(), "k_block_prep_b") == passes
F.fake_capture(0)
assert block(c, p, 512, 16384, 1024) == 0                   # room again: all at once
assert count(kernels(), "k_block_prep_b") == 1
""")


# rows of A that 16-byte loads cannot take (both widths of modulus), and a small
# product over a large modulus: calls that need nothing of the context
FREE = [(65521, 3001, 5003, 40), (2147483647, 3001, 5003, 40), (2147483647, 1024, 1024, 64)]


def test_free_calls_run_under_capture_without_a_call_before(lib):
    fake_cuda.run(f"""
c = context()
base = F.fake_used()
F.fake_capture(1)
for p, m, k, nb in {FREE}:
    F.fake_events()
    assert block(c, p, m, k, nb, stream=CAPTURING) == 0, (p, m, k, nb)
    ks = kernels()
    assert len(ks) == 1 and ks[0].startswith("k_block_cc"), ks
assert F.fake_used() == base
""")


def test_free_calls_share_no_scratch(lib):
    """Each takes its scratch from the pool on its own stream and gives it back;
    the context's buffer is neither used nor grown."""
    fake_cuda.run(f"""
c = context()
base = F.fake_used()
for p, m, k, nb in {FREE}:
    for stream in (0, 16, 32):
        assert block(c, p, m, k, nb, stream=stream) == 0
        ks = kernels()
        assert count(ks, "k_block_tc") >= 1 and count(ks, "k_block_cc") == 0, ks
        assert F.fake_used() == base
assert L.gfp_context_destroy(c) == 0
assert "pool destroyed" in F.fake_events().decode()
""")


def test_free_calls_without_memory_take_the_cuda_cores(lib):
    fake_cuda.run(f"""
for pools in (1, 0):
    F.fake_room(280 << 30)
    F.fake_pools(pools)
    c = context()
    if pools:
        F.fake_room(F.fake_used() + 65536)
    for p, m, k, nb in {FREE}:
        assert block(c, p, m, k, nb) == 0, (p, m, k, nb)
        ks = kernels()
        assert len(ks) == 1 and ks[0].startswith("k_block_cc"), ks
        assert L.gfp_dot(c, 65521, 1024, A, B, C, 0) == 0
        F.fake_events()
""")


def test_wide_free_calls_and_the_other_calls(lib):
    """More columns than the tensor-core launches take; and the calls whose rule is
    the context's workspace still use that and fail to grow it under capture."""
    fake_cuda.run("""
c = context()
assert block(c, 65521, 7, 21, 65535 * 64) == 0
assert count(kernels(), "k_block_tc") == 1
assert block(c, 65521, 7, 21, 65535 * 64 + 1) == 0
assert count(kernels(), "k_block_cc") == 1
base = F.fake_used()
assert block(c, 65521, 4096, 4096, 64) == 0 and F.fake_used() > base
F.fake_events()
F.fake_capture(1)
assert block(c, 65521, 4096, 4096, 64, stream=CAPTURING) == 0
assert count(kernels(), "k_block_tc") == 1
assert block(c, 65521, 8192, 4096, 64, stream=CAPTURING) == g.GFP_ERR_CUDA
""")


def test_reported_error_is_not_reported_again(lib):
    """A call that cannot grow its buffer under capture fails; the calls behind it
    do not fail for it."""
    fake_cuda.run("""
c = context()
for _ in range(2):
    F.fake_capture(1)
    assert block(c, 65521, 4096, 4096, 64, stream=CAPTURING) == g.GFP_ERR_CUDA
    F.fake_capture(0)
    assert L.gfp_dot(c, 65521, 1024, A, B, C, 0) == 0
    assert L.gfp_matvec(c, 65521, 1024, 1024, A, 1024, B, C, 0) == 0
""")


def test_free_calls_beside_a_capture(lib):
    """While another stream is being captured, the first such call of a context
    and the later ones run on the tensor cores, and ask the runtime for nothing it
    refuses then; the thread's capture mode is as before."""
    fake_cuda.run(f"""
c = context()
F.fake_capture(1)
for p, m, k, nb in {FREE}:
    assert block(c, p, m, k, nb) == 0
    assert count(kernels(), "k_block_tc") >= 1
assert F.cudaDeviceSynchronize() != 0
mode = ctypes.c_int(0)
F.cudaThreadExchangeStreamCaptureMode(ctypes.byref(mode))
assert mode.value == 0
""")


# (p, m, k, nb, rows of A padded by, tensor cores): each side of the rules that choose
ROUTES = [(65521, 16384, 8, 200, 1, False), (65521, 16384, 12, 200, 1, False), (65521, 16384, 13, 200, 0, True),
          (65521, 16384, 8, 200, 0, True), (65521, 16384, 1, 1, 0, False), (65521, 64, 64, 64, 1, True),
          (2147483647, 500, 200, 64, 0, False), (2147483647, 500, 1024, 64, 0, True),
          (2147483647, 16384, 200, 200, 1, False), (2147483647, 16384, 1024, 200, 1, True),
          (2147483647, 8192, 8192, 64, 0, True), (67108859, 65536, 64, 512, 0, False),
          (67108859, 256, 16384, 64, 1, True), (100003, 500, 200, 64, 0, True), (100003, 500, 32, 64, 0, False)]


def test_routes_on_each_side_of_the_rules(lib):
    fake_cuda.run(f"""
c = context()
for p, m, k, nb, pad, tc in {ROUTES}:
    assert block(c, p, m, k, nb, lda=k + pad) == 0
    ks = kernels()
    assert (count(ks, "k_block_tc") > 0) == tc and (count(ks, "k_block_cc") == 0) == tc, (p, m, k, nb, pad, ks)
""")
