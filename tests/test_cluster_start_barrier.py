"""A CTA may store into another CTA's shared memory only once that CTA runs, which a cluster-wide barrier
ensures.  A missing barrier shows in a run only when a CTA happens to start late, and then as an undefined
store, so the order is checked in the source: in the pair loop of the cluster form of a demons level the first
statement that stores remotely comes after a barrier of the whole cluster."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1907_05993_gb300", "csrc",
                   "demons_cluster.cuh")


def test_a_cluster_barrier_precedes_the_first_remote_store():
    src = re.sub(r"//[^\n]*", "", open(SRC).read())
    loop = src[src.index("for (int pair ="):]           # what runs: the lambdas that store remotely stand above it
    first = loop[:loop.index("for (int k = 0;")]         # before the iterations: every pair passes through it
    # iteration 0 skips what only later iterations run
    body = loop[len(first):]
    guarded = body[body.index("if (k > 0)"):body.index("float ssd")]
    it0 = first + body.replace(guarded, "", 1)
    store = min(m.start() for m in re.finditer(r"\bxpass\(|\bst_remote\(", it0))
    barrier = it0.find("sync_all();")
    assert 0 <= barrier < store
