"""Orderings that the kernels need and no run can show to be missing, and one
cost that no result shows, read from the sources (comments removed)."""
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


def test_rewritten_stages_are_fenced_before_they_are_handed_back():
    """Images re-made in place are ordinary stores to a stage that a bulk copy
    (the asynchronous proxy) fills next: a proxy fence has to stand between
    them and the arrival that hands the stage back."""
    k = body(source("kg_krylov.cu"), r"k_reorth_dots_int\(")
    store = k.index("img[k * T + e] =")
    back = k.index("mbar_arrive(empty", store)
    assert "proxy_fence(" in k[store:back]
    assert "fence.proxy.async" in body(source("kg_internal.h"), r"void proxy_fence\(")


def test_scalars_are_read_on_the_stream_that_writes_them():
    """The kernels run on non-blocking streams, which a synchronous cudaMemcpy
    (the legacy stream) does not wait for: a status read that way can miss
    what the last steps report."""
    for name in sorted(os.listdir(CSRC)):
        for call in re.findall(r"\bcudaMemcpy\s*\(([^;]*)", source(name)):
            assert not ("DeviceToHost" in call and re.search(r"\bcs\b", call)), (name, call)


def test_no_constant_table_in_a_shared_header():
    """A __constant__ table in a header gives every module that includes it a
    constant bank, which each launch of each of its kernels pays for."""
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".h"):
            assert "__constant__" not in source(name), name
