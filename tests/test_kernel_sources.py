"""What the kernels' sources have to keep to where no run on a GPU shows it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_21624_b200", "csrc")


def kernels(name):
    """The text of each kernel of a source file, from one __global__ to the next."""
    text = open(os.path.join(CSRC, name)).read()
    starts = [m.start() for m in re.finditer(r"__global__", text)] + [len(text)]
    bodies = [text[a:b] for a, b in zip(starts, starts[1:])]
    return {re.search(r"(\w+)\((?:const __grid_constant__|int)", body).group(1): body for body in bodies}


@pytest.mark.parametrize("source", ["k_tc_gemm.cu", "k_tc_attn.cu"])
def test_bulk_stores_and_reductions_are_complete_before_a_block_exits(source):
    # a kernel that hands tiles to bulk copies, itself or through the shared epilogue, waits for the copies and not only for
    # their sources to have been read
    issuing = {k: t for k, t in kernels(source).items() if "bulk_commit_group()" in t or "epilogue_tile<" in t}
    assert issuing
    for k, t in issuing.items():
        assert "bulk_wait_group0()" in t, k
