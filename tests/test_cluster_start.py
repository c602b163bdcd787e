"""The cluster kernel's start: a block may store into another block's shared
memory, or write what the others still copy, only once every block of its
cluster has started and taken its copies.  Read off the source (no GPU: a
kernel without that barrier is not to be run)."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _kernel():
    src = open(os.path.join(ROOT, "paper_0809_2811_gb300", "csrc", "mw_cluster.cuh")).read()
    src = re.sub(r"//[^\n]*", "", src)
    at = src.index("k_cluster(")
    return src[src.index("{", src.index(")", src.index("CluArgs A", at))):]


def test_first_remote_access_follows_an_unconditional_cluster_barrier():
    body = _kernel()
    # stores into other blocks' shared memory, and rank 0's writes of the box's globals
    remote = re.compile(r"clu_flags\(|clu_st\(|clu_rebuild\(|d\.bst\[b\]\.ew\[par\]\[tid\] =|const_cast<Box\*>")
    first = remote.search(body).start()
    before = body[:first]
    barrier = before.rfind("clu_sync();")
    assert barrier >= 0
    # at the kernel's own brace level, so that every thread of every block meets it
    assert before[:barrier].count("{") - before[:barrier].count("}") == 1
    # after the copies of the box, its state and the run's progress
    for copy in ("&S.bx)[k]", "&S.bs)[k]", "&S.I)[k]", "A.prog[b]", "A.mid[b]"):
        assert 0 <= before.find(copy) < barrier, copy
