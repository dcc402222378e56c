"""Source rule (CPU): a bounded wait can end differently for the lanes of a warp (one gives up on the limit while another sees the
phase complete), so a role that runs warp-wide instructions behind it (mma.sync, tcgen05.ld / st, votes) must agree on the
answer first; only a role of one thread, or one that re-joins through bounds of its own, takes the lane's own answer."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_36800_b200", "csrc")


def test_waits_of_the_row_stream_kernel():
    src = open(os.path.join(CSRC, "gemm_row.cu")).read()
    body = src[src.index("bitdelta_gemm_row_kernel("):]
    producer, consumers = body.split("// ------------------------------------------------------------ consumers")
    assert producer.count("wait_bar(") == 1 and "if (lane == 0) {" in producer
    waits = re.findall(r"[^\n]*wait_bar\([^\n]*", consumers)
    assert waits and all("warp_all(" in w for w in waits), waits
