"""Batched dot products at the edges of the persistent kernel's work list: fewer
units than CTAs, as many, more; pairs of one unit (written at once), of several
(one atomic each) and of more than the 65535 units that the packed count holds;
ragged ends of one to three vectors a thread."""
import json

import numpy as np
import pytest
import torch

import gfp_inputs as gi
import oracle
from gpu_util import dev, empty, host

pytestmark = pytest.mark.gpu


def run(lib, ctx, pairs):
    """pairs: (p, n, front): operands start `front` words past an aligned start."""
    xs, ys, descs = [], [], []
    for i, (p, n, front) in enumerate(pairs):
        x, y = gi.uniform(p, n, 94, 2 * i), gi.uniform(p, n, 94, 2 * i + 1)
        xd, yd = dev(x, front), dev(y, front)
        xs.append((p, x, y))
        ys.append((xd, yd))
        descs.append((p, xd, yd, n))
    want = np.array([oracle.dot(p, x, y) if x.size else 0 for p, x, y in xs], np.uint32)
    out = empty(len(pairs))
    plan = lib.BatchPlan(ctx, descs)
    for _ in range(3):   # the scratch returns to zero after each launch
        out.fill_(-1)
        plan.exec(out)
        torch.cuda.synchronize()
        assert np.array_equal(host(out), want)
    plan.close()
    out.fill_(-1)
    lib.gfp_dot_batched(ctx, descs, out)
    torch.cuda.synchronize()
    assert np.array_equal(host(out), want)


@pytest.mark.parametrize("count", [1, 2, 455, 456, 457, 1000])
def test_unit_counts_around_the_grid(lib, ctx, count):
    run(lib, ctx, [((65521, 4294967291, 32749)[i % 3], 1 + 37 * (i % 11), 0) for i in range(count)])


@pytest.mark.parametrize("n", [0, 1, 3, 1023, 1024, 1025, 2047, 2049, 3071, 3073, 4095, 4097, 5119, 7171])
@pytest.mark.parametrize("front", [0, 1])
def test_ragged_ends(lib, ctx, n, front):
    run(lib, ctx, [(p, n, front) for p in (65521, 67108859, 4294967291)])


def test_mixed_one_and_many_units(lib, ctx):
    run(lib, ctx, [(65521, 100, 0), (4294967291, 65536, 0), (2147483647, 65537, 0), (32749, 300001, 0),
                   (67108859, 0, 0), (4294967291, 1 << 20, 0)])


def test_more_units_than_the_packed_count_holds(lib, tmp_path):
    """A plan file with 4096-element work units and one pair of 65537 of them."""
    p, n = 65521, 65536 * 4096 + 5
    path = tmp_path / "plan.json"
    path.write_text(json.dumps({"version": 1, "entries": [{"p": p, "lg_n": 28, "repr": 2, "chunk": 4096}]}))
    c = lib.Context(0)
    try:
        lib.gfp_plan_load(c, str(path))
        x = torch.full((n,), p - 1, dtype=torch.int32, device="cuda")
        y = torch.full((n,), p - 2, dtype=torch.int32, device="cuda")
        out = empty(1)
        plan = lib.BatchPlan(c, [(p, x, y, n)])
        assert plan.info()[0] == 65537
        for _ in range(2):
            out.fill_(-1)
            plan.exec(out)
            torch.cuda.synchronize()
            assert int(host(out)[0]) == 2 * n % p   # (-1)(-2) n
        plan.close()
    finally:
        c.close()
