"""What the compiler says of the kernels: the grouped SIMT kernels keep their
sums in registers (some bytes beside the loop are fine, hundreds are not)."""

import os
import re

import pytest


@pytest.fixture(scope="module")
def info():
    from paper_1608_05265_gb300 import build
    build.build()
    path = os.path.join(build.OUT, "grouped.ptxas")
    return open(path).read()


def test_grouped_simt_kernels_do_not_spill(info):
    found = re.findall(r"Compiling entry function '(\w*grouped_simt_kernel\w*)'.*?(\d+) bytes spill stores, "
                       r"(\d+) bytes spill loads", info, re.S)
    assert len(found) == 24
    assert max(int(stores) for _, stores, _ in found) <= 100, found


def test_splitk_reduction_keeps_its_blocks_on_an_sm():
    """A call in its loop (for exponents that are rarely there) took 128 registers
    a thread and half of the blocks away."""
    from paper_1608_05265_gb300 import build
    build.build()
    text = open(os.path.join(build.OUT, "split.ptxas")).read()
    found = re.findall(r"Compiling entry function '(\w*splitk_reduce_kernel\w*)'.*?Used (\d+) registers", text, re.S)
    assert len(found) == 4  # eight or sixteen (two blocks an SM) loads in flight, each with and without exponents
    assert sorted(int(regs) <= 64 for _, regs in found)[-2:] == [True, True], found
    assert max(int(regs) for _, regs in found) <= 128, found
