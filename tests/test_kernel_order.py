"""Orderings that the kernels need and no run can show to be missing, read from
the sources (comments removed)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1109_1205_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def body(text, head):
    """The braced body after the first match of `head`."""
    at = text.index("{", re.search(head, text).end())
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at:i + 1]
    raise AssertionError(head)


def test_cluster_runs_before_its_shared_memory_is_written():
    """Distributed shared memory may be accessed only once every block of the
    cluster has started, which a cluster barrier in between ensures."""
    k = body(source("kg_small.cu"), r"k_small_step\(")
    barrier = min(i for i in (k.find("cluster_wait("), k.find("cluster_sync(")) if i >= 0)
    assert barrier < k.index("remote_store("), "remote store before the first cluster barrier"
