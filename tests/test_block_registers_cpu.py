"""The tensor-core block kernel hands registers between its roles with
setmaxnreg, whose rules a wrong build breaks by waiting forever rather than by an
error: they are checked here from the source and from ptxas (no GPU needed)."""
import os
import re

import pytest

import fake_cuda
from test_build_cpu import CSRC, ptxas_info


def source():
    text = open(os.path.join(CSRC, "gfp_block.cu")).read()
    return re.sub(r"//[^\n]*", "", text)


def test_each_share_is_set_by_one_instruction_ahead_of_the_roles():
    """The .aligned form wants all warps of a warpgroup at the same instruction.
    The last warpgroup holds several roles, so a share set inside a role's
    branch would be two instructions."""
    src = source()
    kernel = src[src.index("k_block_tc(const __grid_constant__ Args a)"):src.index("struct PrepB")]
    uses = [(m.start(), m.group(1)) for m in re.finditer(r"regs_(?:inc|dec)<(\w+)>", kernel)]
    assert sorted(name for _, name in uses) == ["REGS_CONV", "REGS_EPI", "REGS_MMA"]
    first_role = kernel.index("ALoads<MODE, PRE> ld")
    assert all(at < first_role for at, _ in uses)


def test_kernels_compile_to_the_registers_that_are_shared_out():
    """setmaxnreg.inc draws on what the block was launched with: fewer registers a
    thread than the shares add up to would leave the converters waiting forever,
    more would not fit one block of 896 threads."""
    launch = int(re.search(r"REGS_LAUNCH = (\d+)", source()).group(1))
    regs, spills = ptxas_info("gfp_block.cu")
    tc = {k: v for k, v in regs.items() if "k_block_tc" in k}
    assert len(tc) == 5 and set(tc.values()) == {launch}, tc
    assert launch * 896 <= 65536
    assert all(spills[k] == 0 for k in tc), spills


@pytest.mark.parametrize("regs,launched", [(72, True), (64, False), (80, False)])
def test_other_register_counts_are_refused_before_the_launch(lib, regs, launched):
    fake_cuda.run(f"""
F.fake_regs({regs})
c = context()
for p in (65521, 65521, 2147483647):
    st = block(c, p, 4096, 4096, 64)
    assert st == (g.GFP_OK if {launched} else g.GFP_ERR_CUDA), st
    assert (count(kernels(), "k_block_tc") > 0) == {launched}
""")
