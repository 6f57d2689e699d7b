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
        # `done` counts the answers waited for: n when request n is made, n + 1 when its answer is read
        assert re.findall(r"clc_request\((.*), bar_clc\)", body) == ["clc + (tclc.done & 1)"]
        assert re.findall(r"clc_answer\((.*)\) : -1", body) == ["clc + ((tclc.done & 1) ^ 1)"]
        taken = body[body.index("auto taken"):]
        assert taken.index("track_wait_all(bar_clc, tclc)") < taken.index("clc_answer")
