"""Block products by the scratch they have: B's tiles for one residue modulus at a
time where those of all would be too large."""
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
