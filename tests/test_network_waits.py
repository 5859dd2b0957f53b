"""The network kernels' bounded waits (read from the source: a wait that runs
out cannot be staged lane by lane).  A wait that each lane decides for itself
may end the loop for some lanes of a warp only, and the others would run into
the warp-wide tcgen05 instructions behind it without them; so it is for
sections that a single lane runs, and every other role waits as a warp."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2012_14707_gb300", "csrc", "lbm_net_tc.cu")


def calls_with_blocks(text, name):
    """For each call of `name`: the headers of the blocks around it, outermost first."""
    text = re.sub(r"//[^\n]*", "", text)
    text = re.sub(r'"(\\.|[^"\\])*"', '""', text)
    stack, start, out = [], 0, []
    call = re.compile(r"\b" + name + r"\(")
    for i, ch in enumerate(text):
        if ch == "{":
            stack.append(" ".join(text[start:i].split()))
            start = i + 1
        elif ch == "}":
            stack.pop()
            start = i + 1
        elif ch == ";":
            start = i + 1
        elif ch == name[0] and call.match(text, i) and not text[i - 1].isalnum() and text[i - 1] != "_":
            if text[start:i].split()[-2:-1] != ["__forceinline__"]:  # its definition
                out.append(stack + [" ".join(text[start:i].split())])
    return out


def test_lane_waits_only_where_one_lane_runs():
    text = open(SRC).read()
    names = set(re.findall(r"\b(mbar_wait\w*)\(", text))
    collective = {"mbar_wait_warp"}
    assert "__all_sync(0xFFFFFFFFu" in text.split("bool mbar_wait_warp(")[1].split("}")[0]
    found = 0
    for name in names - collective:
        for blocks in calls_with_blocks(text, name):
            found += 1
            inside = any("bool mbar_wait_warp(" in b for b in blocks)
            single = any(b.endswith("if (lane == 0)") for b in blocks)
            assert inside or single, (name, blocks[-3:])
    assert found


def test_ring_of_weights_waits_after_the_kernel_before():
    """The weights are copied without waiting for the stream's earlier kernel,
    but a wait for the MMAs to free a block has a limit, and no MMA runs before
    that kernel ends: it may take longer than the limit."""
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    kernel = text.split("conv_halo_tc(const __grid_constant__ ConvDev a) {")[1]
    role = kernel.split("if (warp == 0) {")[1].split("} else if (warp == 1)")[0]
    before = role.split("&empty_b[st]")[0]
    assert re.search(r"if \(issued == a\.stages_b\) chain_wait\(\);", before)
