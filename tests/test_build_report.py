"""What ptxas says of the kernels that the build made (no GPU needed)."""
import os
import re

import pytest

from paper_2504_03702_b200 import build


def frames(source):
    """{function: (bytes of stack, bytes spilled)} of a source's report."""
    name, out = None, {}
    for line in open(build.report(source)):
        m = re.search(r"(?:Compiling entry function|Function properties for) '?([^' ]+)", line)
        if m:
            name = m.group(1).strip()
        m = re.search(r"(\d+) bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads", line)
        if m:
            out[name] = (int(m.group(1)), int(m.group(2)) + int(m.group(3)))
    return out


@pytest.mark.parametrize("source", ["whole", "whole_admit", "halves", "halves_admit", "rounded", "rounded_admit"])
def test_the_deciding_loop_keeps_nothing_on_the_stack(source):
    """Its rows' keys are registers; a part of it that is called instead of inlined takes them by reference, hence through memory (frames of 992
    to 2,032 bytes, and batches twice as long)."""
    build.build()
    found = frames(os.path.join(build.CSRC, f"route_summary_{source}.cu"))
    kernels = {k: v for k, v in found.items() if "pre_route_summaries" in k and "lambda" not in k and "rs_" not in k}
    assert len(kernels) == (5 if "halves" in source else 6)      # (one per number of rows held; exact fractions begin beyond the smallest)
    assert all(v == (0, 0) for v in kernels.values()), kernels
    assert not [k for k in found if "rs_decide_loop" in k], "a part of the deciding loop is a function of its own"
