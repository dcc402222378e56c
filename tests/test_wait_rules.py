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


def test_waits_of_the_several_tenants_roles():
    # (decode: tcgen05.st behind the sign words' and the operand buffer's wait; epilogue: tcgen05.ld behind the accumulators')
    src = open(os.path.join(CSRC, "gemm_tc.cu")).read()
    branch = src[src.index("// warp (grp, quad): the tenants j = grp, grp+2, ..., one buffer of the group's ring each"):]
    assert re.search(r"wait_bar\(", branch[:branch.index("tmem_st32")]) and "warp_all(wait_bar(aempty_g" in branch[:branch.index("tmem_st32")]
    for wait in (r"wait_bar\(smem_u32\(&ctl->bfull\[bslot\]\), bphase, abort_flag, 6\);", r"wait_bar\(smem_u32\(&ctl->accfull\), accphase, abort_flag, 8\);"):
        assert re.search(wait + r"\s+if constexpr \(kGrouped\) ok = warp_all\(ok\);", src), wait


def test_waits_of_the_compress_kernel():
    # (the producer is one thread; the consumers' shuffles and their arrivals come behind a wait whose answer the warp shares)
    src = open(os.path.join(CSRC, "compress.cu")).read()
    body = src[src.index("compress_kernel("):src.index("__global__ void compress_finish_kernel(")]
    producer, consumers = body[:body.index("// Lane l's 64 bytes of a tile")], body[body.index("// Lane l's 64 bytes of a tile"):]
    assert producer.count("wait_bar(") == 1 and producer.index("if (lane == 0) {") < producer.index("wait_bar(")
    waits = re.findall(r"[^\n]*wait_bar\([^\n]*", consumers)
    assert len(waits) == 1 and "ok = warp_all(ok && wait_bar(" in waits[0], waits
