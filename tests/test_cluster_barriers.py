"""Distributed shared memory: a CTA may store into another's shared memory only once a cluster barrier has shown that
the other has begun, and must not end while stores into its own are on their way.  A violation is a race that a run
does not reliably show, so the order is checked in the source.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_02718_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def _body(src, name):
    """The braces of the function `name`'s definition."""
    for m in re.finditer(r"\b%s\(" % name, src):
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(src[i], 0)
            i += 1
        if src[i:].lstrip().startswith("{"):
            start = i = src.index("{", i)
            depth = 0
            while True:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
                if depth == 0:
                    return src[start:i]
    raise AssertionError(name)


def test_the_cluster_has_begun_before_the_first_remote_store():
    body = _body(_source("solvers.cu"), "k_cg_small")
    first = body.index("cluster_sum(")
    wait = max(body.rfind("cl.barrier_wait(", 0, first), body.rfind("cl.sync(", 0, first))
    assert wait >= 0
    if "cl.barrier_wait(" in body:
        arrive = body.index("cl.barrier_arrive(")
        assert arrive < wait and body.count("barrier_arrive(") == body.count("barrier_wait(") == 1
        assert "return" not in body[arrive:wait]  # every thread that arrives waits


def test_remote_stores_are_followed_by_a_cluster_barrier():
    src = _source("solvers.cu")
    assert src.count("map_shared_rank") == 1  # the one place that reaches another CTA's memory
    body = _body(src, "cluster_sum")
    assert body.index("map_shared_rank") < body.index("cl.sync(")


def test_the_cluster_kernel_runs_only_where_a_cluster_fits():
    """A cluster of 16 CTAs may not fit where a GPU is shared out; its launch would fail there.  The solver asks first
    and otherwise takes the kernels that need no cluster (which tests/test_gpu_cg_small.py covers, just above the
    limit on the length)."""
    src = _source("solvers.cu")
    fits = _body(src, "cg_small_fits")
    assert "cudaOccupancyMaxActiveClusters(" in fits
    run = _body(src, "run_cg")
    flag = re.search(r"const bool small = ([^;]*);", run).group(1)
    assert "cg_small_fits" in flag
    assert run.index("if (small)") < run.index("k_cg_small<T><<<")  # its one launch, under that flag
    assert src.count("k_cg_small<T><<<") == 1


def test_no_other_kernel_reaches_a_peers_shared_memory():
    for name in sorted(os.listdir(CSRC)):
        if name != "solvers.cu":
            assert not re.search(r"map_shared_rank|\bmapa\b|__cluster_dims__", _source(name)), name
