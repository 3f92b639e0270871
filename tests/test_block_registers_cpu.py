"""The tensor-core block kernel hands registers between its roles with
setmaxnreg, whose rules a wrong build breaks by waiting forever rather than by an
error: they are checked here from the source and from ptxas (no GPU needed)."""
import os
import re

from test_build_cpu import CSRC


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
