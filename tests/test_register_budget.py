"""Registers of the line-walk kernels, from the build's ptxas log: the block
counts that their launch bounds ask for fit an SM's 65,536 registers, and no
kernel that runs outside debug solves keeps values in local memory."""
import os
import re

import pytest

from paper_2305_04403_gb300 import build as B

# kernel: most registers a thread for its blocks of 128 per SM (multiples of 8)
BUDGET = {"k_dl_linesILb0ELb0ELb0EE": 80, "k_dl_linesILb0ELb0ELb1EE": 80, "k_nd_linesILb0EE": 72,
          "k_fwd_lines": 96, "k_batch_linesILi1EE": 80, "k_batch_linesILi2EE": 80,
          "k_batch_linesILi4EE": 80, "k_dl_groupsILb0EE": 80, "k_dl_groupsILb1EE": 80,
          "k_nd_groups": 80, "k_fwd_groups": 80, "k_sl_walks_ffILb0EE": 72,
          "k_sl_walks_risILb0EE": 72}


@pytest.fixture(scope="module")
def functions():
    B.build()
    out = {}
    for block in open(os.path.join(B.OUT, "ptxas.log")).read().split("Function properties for ")[1:]:
        regs = re.search(r"Used (\d+) registers", block.split("Compiling entry function")[0])
        if regs:
            spill = int(re.search(r"(\d+) bytes spill stores", block).group(1))
            out[block.split()[0]] = (int(regs.group(1)), spill)
    return out


@pytest.mark.parametrize("kernel", sorted(BUDGET))
def test_line_walks(functions, kernel):
    found = [v for k, v in functions.items() if kernel in k]
    assert len(found) == 1, kernel
    assert found[0][0] <= BUDGET[kernel] and found[0][1] == 0, found
