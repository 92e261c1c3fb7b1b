"""What a wait that gives up may still do in the one-kernel score of short caches, whose CTAs write into one another's shared memory.  Making a
wait give up on a GPU is not an option for a test, so the rules are held against the kernel's source: nothing is announced after a failure,
and a CTA in which a wait failed leaves only after the cluster's others have issued everything and all of it has landed."""
import os
import re

from paper_2510_07651_b200 import build


def _kernel():
    text = open(os.path.join(build.CSRC, "score_tc.cu")).read()
    body = text[text.index("tc_short_kernel(const __grid_constant__"):text.index("// ---- host side")]
    return re.sub(r"//[^\n]*", "", body)


def test_nothing_is_announced_after_a_failed_wait():
    body = _kernel()
    arrivals = re.findall(r"[^\n;{}]*\b(?:mbar_arrive|arrive_at_cta)\(", body)
    assert len(arrivals) == 2 and all("none_failed() &&" in a for a in arrivals)
    assert re.search(r"none_failed = [^;]*;[^;]*__all_sync\(0xffffffffu, !failed\)", body)
    assert re.search(r"if \(wait\(SH_STAGED, __LINE__\)[^;{}]*\)\s*for \([^;]*;[^;]*;[^)]*\)\s*copy_to_cta\(", body)
    assert re.search(r"wait\(SH_RX, __LINE__\)\) \{(?:(?!\n        \}).)*st_cluster2\(", body, re.S)


def test_a_cta_with_a_failed_wait_outlives_what_is_under_way():
    end = _kernel()
    end = end[end.rindex("atomicCAS(p.status"):]
    drained = re.search(r"if \(__syncthreads_or\(failed\)\) \{\s*cluster_arrive\(\); cluster_wait\(\);(.*)cluster_arrive\(\); cluster_wait\(\);\s*\}", end, re.S)
    assert drained and all(f"mbar_wait(bar({b}), 0)" in drained[1] for b in ("SH_RX", "SH_QK", "SH_V", "SH_DRAIN"))
    assert drained.end() < end.index("tcgen05.dealloc")
