"""The clustered walk's use of distributed shared memory, read from its source: a CTA may store into
another CTA of its cluster only after a cluster barrier has shown that the other one runs, and may
not store after the last barrier (the other one may have ended).  A missing barrier shows in no
output, so the order of the source is what can be checked."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_04336_gb300", "csrc")


def walk_kernel_body():
    text = open(os.path.join(CSRC, "kernels_impl.cuh")).read()
    text = re.sub(r"//[^\n]*", "", text)
    start = text.index("walk_kernel(const EventDev*")
    depth, i = 0, text.index("{", start)
    first = i
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[first:i + 1]
        i += 1


def test_cluster_barrier_before_the_first_remote_store():
    body = walk_kernel_body()
    sync, loop = body.index("cluster.sync()"), body.index("while (t < n_steps)")
    assert body.count("return;", 0, loop) == 1        # of finished walkers: every rank of one returns
    assert body.index("return;") < sync < loop
    assert sync < body.index("map_shared_rank")


def test_cluster_barrier_after_the_last_remote_store_of_a_round():
    body = walk_kernel_body()
    last = body.rindex("map_shared_rank")
    stores = [m.start() for m in re.finditer(r"store_total\(", body)]
    assert max(stores + [last]) < body.rindex("cluster.sync()")
