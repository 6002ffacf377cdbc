"""What can be seen without a GPU of how the kernels were written and built: ptxas' report, and the order of a hand-over in the source."""
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


def body(text, opening):
    """From `opening` to the brace that closes it."""
    at = text.index(opening)
    depth, end = 0, at
    for end in range(text.index("{", at), len(text)):
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        if depth == 0:
            break
    return text[at:end + 1]


def test_the_words_of_a_list_are_read_with_its_number():
    """The list block writes them from another SM, and nothing orders them behind the word that says a list is there.  No run shows a word that is read too
    early (shared memory is read in order where it is compiled so), so the source is looked at: the list's words are read by relaxed loads alone, the
    deciding warp takes none before each has the list's number, and the io warp, which does not look for it, no row that there is not."""
    text = open(os.path.join(build.CSRC, "route_summary.cuh")).read()
    code = "\n".join(line.split("//")[0] for line in text.splitlines())
    for word in ("list_row[", "list_base["):
        reads = [line for line in code.splitlines() if "sh." + word in line and "other_smem" not in line and not re.search(r"\] = 0;", line)]
        assert reads and all("ld_relaxed_cluster(&sh." + word in line for line in reads), reads
    take = body(code, "auto next_list = [&](unsigned int e) {")
    assert take.index("there = K::of_list(") < take.index("there &= of_list(word[k]") < take.index("there &= of_list(half[x]") < take.index("RS_LIST_NOBODY")
    asks, builds = body(code, "auto ask_for_list = [&]() {"), body(code, "void rs_build_lists(")
    assert "st_release(&sh.list_free" in asks and "st_release_cluster(other_smem(&sh.list_free" in body(code, "void rs_pass_on(")
    assert builds.index("told(&sh.lists_wanted") < builds.index("told(&sh.list_free") < builds.index("st_cluster(at_list")
    touch = body(code, "void rs_io_loop(")
    assert touch.index("if (w < (unsigned int)a.I)") < touch.index("touch_row(a.near")


def test_a_batch_is_given_up_by_the_whole_block():
    """The list block, on another SM, may store the word that says a wait was abandoned until it is told to leave: the routing block's threads branch on one common
    look at it (a barrier follows that branch), and the status of the batch is that look's."""
    text = open(os.path.join(build.CSRC, "route_summary.cuh")).read()
    code = "\n".join(line.split("//")[0] for line in text.splitlines())
    route = body(code, "__device__ __forceinline__ bool rs_route(")
    assert [line.strip() for line in route.splitlines() if "ctl.w" in line] == ["const bool lost = __syncthreads_or(ld_volatile(&sh.ctl.w) != 0) != 0;"]
    assert "ctl.w" not in body(code, "pre_route_summaries(const __grid_constant__ RouteSumArgs a) {")
