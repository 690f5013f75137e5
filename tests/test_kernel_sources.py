"""Rules of the kernels that no run shows: they concern launches whose bounded waits have given up, or a later change of a launch."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_17560_b200", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def test_a_pair_that_gave_up_orders_its_arrivals():
    """The pair GEMMs' last cluster barrier orders no memory, which is sound only while every arrival sent to the leader is one it
    waits for.  All four epilogues fence where they give a wait up, and the barrier acquires."""
    kernel = source("a3_gemm_persistent.cu").split("pair_t_kernel(", 1)[1].split("bool swiglu_pair_usable", 1)[0]
    assert re.search(r"give_up = \[\] \{ asm volatile\(\"fence.acq_rel.cluster;\"", kernel)
    left = re.findall(r"if \(!ep_ok\[0\]\) \{\s*(.*?)\s*\}", kernel, flags=re.S)
    assert len(left) == 4 == len(re.findall(r"ep_ok\[0\] = mbar_wait", kernel))
    assert all(re.match(r"give_up\(\);\s*(break|return false);", body) for body in left)
    barrier = source("a3_tc.cuh").split("cluster_sync_relaxed()", 1)[1].split("}", 1)[0]
    assert "arrive.relaxed" in barrier and "wait.acquire" in barrier


def test_launches_that_others_run_beside_are_ordinary():
    """rerotate_kernel and clear_ticket_kernel let their successors start early, which write before they wait: sound only because these
    two waited for everything before them.  Only rerotate itself says whether there is such a launch to run beside."""
    for name, kernel in (("a3_stream_kernels.cu", "rerotate_kernel"), ("a3_first_token.cu", "clear_ticket_kernel")):
        text = source(name)
        assert re.search(kernel + r"(<\w+, \w+>)?<<<", text)
        assert not re.search(r"launch_pdl(_cluster)?\([^;]*" + kernel, text)
    ticket = source("a3_first_token.cu").split("clear_ticket_kernel<<<")[1]
    assert ticket.split("launch_pdl(")[0].count(";") == 2  # the launch and its check, nothing queued in between
    for call in re.findall(r"enter_rows\([^;]*;", source("a3_api.cu")):
        last = call.rsplit(",", 1)[1].strip(" \n);")
        assert last in ("st", "recovering", "i == 0 && recovering"), last
