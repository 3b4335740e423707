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


def test_last_ctas_fence_before_their_barrier():
    """Every count of CTAs goes through the helper that fences on both sides, and a CTA's barrier follows it; the only
    other add to a counter in global memory is the layer step's (above)."""
    helper = _code("common.cuh")
    body = helper[helper.index("bool arrive_is_last("):]
    body = body[:body.index("\n}")]
    assert re.search(r"__threadfence\(\);.*atomicAdd\(.*if \(last\) __threadfence\(\);", body, flags=re.S)
    calls = 0
    for name in sorted(os.listdir(CSRC)):
        code = _code(name)
        for add in re.finditer(r"atomicAdd\(([^,]*),", code):
            at = add.group(1).strip()
            assert at.startswith("&s_") or (name, at) in (("common.cuh", "cnt"), ("decode_step.cu", "&ws.cnt[seg]")), \
                (name, at)   # &s_...: shared memory
        for call in re.finditer(r"= arrive_is_last\([^;]*\);\s*\}\s*(\w+\(\);)", code):
            assert call.group(1) == "__syncthreads();", name
            calls += 1
        assert code.count("= arrive_is_last(") == len(re.findall(r"= arrive_is_last\([^;]*\);\s*\}\s*__syncthreads", code))
    assert calls == 6
