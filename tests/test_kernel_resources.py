"""Registers of the kernels whose launch bounds differ by form, from the
assembler's report of the build."""
import os
import re

from paper_1411_2087_gb300 import build


def kernels(unit, name):
    """{mangled entry: registers} of the kernels `name` in one translation unit."""
    build.build()
    text = open(os.path.join(build.BUILD, unit + ".ptxas")).read()
    found = re.findall(r"Compiling entry function '(\w+)'.*?Used (\d+) registers", text, flags=re.S)
    return {e: int(r) for e, r in found if f"{len(name)}{name}I" in e}


def test_net_mid_blocks_by_form():
    """128-thread blocks: six per SM leave 80 registers, seven 72.  The
    double-float forms, and FP64 on FP32 links, use what seven would deny."""
    regs = kernels("kernels_netpath", "net_mid_kernel")
    assert len(regs) == 13
    for e, r in regs.items():
        six = "kernelILi3E" in e or "kernelILi0E6float2" in e
        assert 72 < r <= 80 if six else r <= 72, (e, r)
