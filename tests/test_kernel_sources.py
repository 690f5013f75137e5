"""Rules of the kernels that no run shows: they concern launches whose bounded waits have given up, or a later change of a launch."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_17560_b200", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def test_a_pair_that_gave_up_leaves_through_a_releasing_barrier():
    """The pair GEMMs' last cluster barrier orders no memory, which is sound only while every arrival sent to the leader is one it
    waits for.  All four epilogues report a wait that gave up, and these warps take the barrier that does order."""
    kernel = source("a3_gemm_persistent.cu").split("pair_t_kernel(", 1)[1].split("bool swiglu_pair_usable", 1)[0]
    last = [line.strip() for line in kernel.splitlines() if "cluster_sync_" in line][-2:]
    assert last == ["if (__any_sync(0xffffffffu, gave_up)) cluster_sync_all();", "else cluster_sync_relaxed();"]
    assert kernel.count("cluster_sync_relaxed") == 1
    assert len(re.findall(r"gave_up = !sp_with_chunk<", kernel)) == 3 == len(re.findall(r"sp_with_chunk<", kernel))
    assert len(re.findall(r"if \(!ep_ok\[0\]\) return false;", kernel)) == 3
    assert re.search(r"if \(!ep_ok\[0\]\) \{\s*gave_up = true;\s*break;", kernel)
