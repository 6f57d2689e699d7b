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
