"""Ordering that the kernels' shared memory depends on, read from their sources (CPU only): a
missing barrier of this kind shows on a GPU only when the timing is unlucky."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_14898_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as fh:
        return "\n".join(line.split("//", 1)[0] for line in fh)


def _kernel(src, name):
    """Body of the function `name`: its text up to the closing brace in the first column."""
    m = re.search(r"\b%s\(" % name, src)
    return src[m.start():src.index("\n}", m.start())]


def test_cluster_started_before_peer_shared_memory():
    """The cross-entropy cluster writes its peers' shared memory only behind a cluster barrier
    (outside of the row loop, so on every path): before it a peer may not have started."""
    body = _kernel(_code("client.cu"), "ce_cluster_kernel")
    head = body[:body.index("for (int row")]
    assert "st_cluster_f2" in body and "st_cluster_f2" not in head
    assert re.search(r"cluster_arrive\(\)[\s\S]*cluster_wait\(\)|cluster_sync\(\)", head)


def test_launch_control_answers_alternate():
    """Attention backward: a cluster launch control request never targets the shared memory that
    other warps may still be reading the previous answer from.  Request n goes to slot n % 2 and its
    answer is read from there; the CTA-wide wait for answer n + 1, which every thread reaches only
    after reading answer n, lies before request n + 2."""
    src = _code("attention_bwd_tc.cu")
    for name in ("attn_bwd_dkv_tc_kernel", "attn_bwd_dq_tc_kernel"):
        body = _kernel(src, name)
        slots = int(re.search(r"holder = reinterpret_cast<uint32_t\*>\(bars \+ (\d+)\)", body).group(1)) - \
            int(re.search(r"clc = reinterpret_cast<uint4\*>\(bars \+ (\d+)\)", body).group(1))
        assert slots == 4  # two answers of 16 bytes
        # the parity of the answers waited for: n % 2 when request n is made, (n + 1) % 2 when its answer is read
        assert re.findall(r"clc_request\((.*), bars \+ B_CLC\)", body) == ["clc + tr.parity(B_CLC)"]
        assert re.findall(r"wait_all\(B_CLC, .*?\) \? clc_answer\((.*)\) : -1", body) == ["clc + (tr.parity(B_CLC) ^ 1)"]


def test_products_wait_for_the_readers_of_their_columns():
    """Attention: a score product whose TMEM columns hold an operand of a product in flight is issued
    behind a wait for it (PTX orders only products of one shape and accumulator).  Forward: the next
    S over the P that P V reads; backward: S^T over the P^T that dV reads, dP^T over the dS^T that
    dK reads (behind the next S^T, committed after dK); dQ's dS has columns of its own."""
    fwd = _kernel(_code("attention_tc.cu"), "attn_fwd_tc_kernel")
    p_over_s = re.search(r"T_P = HD == 64 \? 192 : 0;", fwd)
    assert p_over_s and "pv_waited = T_P == 0;" in fwd
    assert "if (warp == 0 && (!pv_waited || mbar_wait_warp(bars + B_PV, tr.parity(B_PV)))) score();" in fwd
    src = _code("attention_bwd_tc.cu")
    dkv = _kernel(src, "attn_bwd_dkv_tc_kernel")
    loop = dkv[dkv.index("for (int it = w.it0"):]
    # in the loop: dP^T behind the CTA-wide wait for S^T, S^T behind the wait for dV
    assert loop.index("wait_all(ONE ? B_DP : B_S,") < loop.index("scores(b, 1)") < loop.index("scores(1 - b, 0)")
    assert loop.index("mbar_wait_warp(bars + B_DV, tr.parity(B_DV))") < loop.index("scores(1 - b, 0)")
    assert len(re.findall(r"\bscores\(", loop)) == 2
    dq = _kernel(src, "attn_bwd_dq_tc_kernel")
    assert "T_DS = 256 + HD;" in dq
    assert re.findall(r"umma_bf16_ts\(tmem \+ 256, (.*?), bk", dq) == ["tmem + T_DS + 8 * kk"]


def test_given_up_waits_end_behind_every_product():
    """Attention: when a wait gave up, the issuing warp commits once more and waits for it before the
    CTA frees its TMEM, so that no product (committed before or not) is still at work on it."""
    kernels = [("attention_tc.cu", "attn_fwd_tc_kernel"), ("attention_bwd_tc.cu", "attn_bwd_dkv_tc_kernel"),
               ("attention_bwd_tc.cu", "attn_bwd_dq_tc_kernel")]
    for name, kernel in kernels:
        body = _kernel(_code(name), kernel)
        end = re.search(r"if \(!ok && warp == 0\) \{\s*if \(elect_one\(\)\) umma_commit\(bars \+ B_END\);\s*"
                        r"mbar_wait_warp\(bars \+ B_END, 0\);\s*\}", body)
        assert end and max(m.start() for m in re.finditer(r"umma_bf16", body)) < end.start() < body.index("tmem_dealloc")


def test_warp_wide_loops_agree_on_an_expired_wait():
    """GEMM epilogues: their loops hold warp-wide TMEM reads, so a wait that gives up does so for the
    whole warp; a lane alone must not leave the loop."""
    src = _code("gemm_tc.cuh")
    for name in ("epilogue_loop", "adamw_epilogue", "f32_epilogue"):
        body = _kernel(src, name)
        waits = re.findall(r"if \(!(.*?mbar_wait\w*)\(", body)
        assert waits and all(w in ("mbar_wait_warp", "__all_sync(0xffffffffu, mbar_wait") for w in waits), name
