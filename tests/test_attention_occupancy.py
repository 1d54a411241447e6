"""The attention kernel of many tiles is chosen because two of its CTAs share an SM: its launch bound has to ask for that
(a compiler that is free to take more registers would undo it without a word).  Shared memory is asserted when the library
is compiled."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_15618_b200", "csrc")


def test_launch_bound_asks_for_the_ctas_the_ring_depth_was_chosen_for():
    text = open(os.path.join(CSRC, "fm_attention.cuh")).read()
    bound = re.search(r"__launch_bounds__\(([^()]*)\)\s*attn_stream_kernel", text).group(1)
    assert bound.split(",")[-1].strip().endswith("::CTAS"), bound
    host = open(os.path.join(CSRC, "flashmesh.cu")).read()
    depths = {int(two is not None and two != ""): set() for two in ("", "if")}
    for two, st in re.findall(r"(if \(two\) |else )launch_pdl\(c, one, attn_stream_kernel<\d+, \d+, \d+, (\d+)>", host):
        depths[int(two.startswith("if"))].add(int(st))
    ctas = re.search(r"CTAS = STAGES <= (\d+) \? 2 : 1", text)
    assert depths[1] and max(depths[1]) <= int(ctas.group(1)) < min(depths[0])
    assert re.search(r"static_assert\(CTAS \* \(BYTES \+ 1024\) <= 228 \* 1024", text)
