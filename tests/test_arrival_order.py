"""Work handed over by counting arrivals: a thread that finds itself the last adds relaxed, so before the barrier that
passes the others' results on to its warp or CTA it has to fence (a fence by the readers, which counted nothing, orders
nothing).  No run can be made to fail without it, so the order is read off the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_27233_gb300", "csrc")


def _code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def test_layer_step_fences_between_its_counts_and_the_merge():
    code = _code("decode_step.cu")
    counted = code.index("atomicAdd(&ws.cnt[seg], 1)")
    assert "__threadfence();" in code[:counted][-400:]      # the partials, before they are counted
    reads = code.index("merge_pieces(sp.o", counted)
    between = code[code.index("s_pend[warp][slot] = seg", counted):reads]
    fence = re.search(r"if \(lane == 0 &&[^;]*\) __threadfence\(\);\s*__syncwarp\(\);", between)
    assert fence, "lane 0 counts: it fences, then the warp's barrier hands the partials on"
    # and the CTA's barrier stands between that fence and the merges that all warps share
    assert code.index("__syncthreads_or(shared)", counted) < code.index("merge_pieces(sp.o, wa", counted)
