"""Instructions of the prefill kernel that a whole warp issues together (.aligned):
after a branch that only some lanes take, a __syncwarp comes first.  Diverged
lanes are a fault that no run is sure to show, so this reads the source."""
import os
import re

PREFILL = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                       "paper_2609_17475_gb300", "csrc", "prefill.cu")
SOURCE = re.sub(r"//[^\n]*", "", open(PREFILL).read())


def _between(start, end):
    at = SOURCE.index(start)
    return SOURCE[at:SOURCE.index(end, at)]


def test_lanes_meet_before_the_allocation():
    assert _between("if (threadIdx.x == 0) {\n    for (int i = 0; i < 4", "tc::alloc2(").rstrip() \
        .endswith("__syncwarp();\n  if (warp == 0)")


def test_lanes_meet_before_the_register_split():
    after = _between("tc::arrive_cluster(q_full, 0);", "tc::setmaxnreg_dec<R::MMA_REGS>")
    assert re.search(r"\}\s*__syncwarp\(\);\s*if \(warp < R::DQ0\) \{\s*$", after), after


def test_lanes_meet_after_each_tile_and_store():
    assert re.search(r"if \(lane == 0\) tc::arrive_cluster\(&p_full\[j & 3\], 0\);\s*__syncwarp\(\);",
                     SOURCE)
    assert re.search(r"\(orow \+ c0 \+ 8 \* k\) = w;\s*\}\s*\}\s*__syncwarp\(\);", SOURCE)


def test_lanes_meet_before_the_last_cluster_barrier():
    assert re.search(r"__syncthreads\(\);\s*__syncwarp\(\);\s*tc::cluster_sync\(\);\s*"
                     r"if \(warp == 0\) \{\s*tc::fence_after\(\);\s*tc::dealloc2", SOURCE)
