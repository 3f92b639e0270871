"""Device memory of the block products' host code, against a stand-in for the CUDA
runtime (no GPU needed): what is asked for, and what a failed allocation leaves."""
import fake_cuda


def test_smaller_buffer_after_a_failed_allocation(lib):
    """A context's buffer is asked for at the size of its largest parts; where that
    does not fit, this product's parts alone do, and the product runs to its end."""
    for p, last in ((65521, "k_block_finish"), (2147483647, "k_block_crt")):
        fake_cuda.run(f"""
c = context()
assert block(c, {p}, 64, 4194304, 64) == 0                  # large tiles of B
assert F.fake_used() > 1 << 30
F.fake_room(F.fake_used() + (64 << 20))
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
