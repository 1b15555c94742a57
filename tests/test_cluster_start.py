"""The single-launch cluster transform writes other CTAs' shared memory. That is defined only once
those CTAs have started, so the kernel arrives at a cluster barrier as it begins and waits on it
before its first remote store. A missing wait shows in no result as long as the CTAs happen to start
together, so the order is checked in the source."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_00546_gb300", "csrc",
                   "ntt_kernels.cuh")


@pytest.fixture(scope="module")
def code():
    return re.sub(r"//[^\n]*", "", open(SRC).read())


def _function(code, name):
    """The text from a function's name to the end of its body."""
    start = re.search(r"\b%s\([^;{]*\)\s*\{" % name, code)
    depth, i = 1, start.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(code[i], 0)
        i += 1
    return code[start.end(): i]


def _barriers(code, ptx):
    """Names of the functions that issue the instruction."""
    return re.findall(r"(\w+)\(\)\s*\{\s*asm volatile\(\"%s" % re.escape(ptx), code)


def test_remote_stores_wait_for_the_cluster_to_have_started(code):
    arrive, = _barriers(code, "barrier.cluster.arrive")
    wait, = _barriers(code, "barrier.cluster.wait")
    assert _function(code, "k_ntt_cluster").split(";")[0].strip() == arrive + "()"
    assert code.count("map_shared_rank") == 2
    forward, inverse = _function(code, "ntt_cluster_body").split("} else {")
    for direction in (forward, inverse):
        first, rest = direction.split("map_shared_rank")   # one set of remote stores a direction
        assert first.count(wait + "()") == 1 and arrive not in direction
        assert "cl.sync()" not in first and "cl.sync()" in rest   # the data barrier follows
