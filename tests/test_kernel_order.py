"""Orderings between threads and CTAs that no run can show to be missing (it
would work until the day it does not): checked on the kernels' source, with
comments removed."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_02464_gb300", "csrc")


def _source(name):
    src = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)


def _body(src, signature):
    """The braces that follow `signature` (a definition that occurs once)."""
    assert src.count(signature) == 1, signature
    i = src.index("{", src.index(signature))
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth == 0:
            return src[i:j + 1]
        j += 1


def test_one_launch_stepping_waits_for_its_cluster_before_the_first_remote_store():
    """Another CTA's shared memory may be accessed only after a cluster
    barrier has shown that the CTA runs."""
    body = _body(_source("weno_run1d.cuh"), "k_run1d(Run1DArgs r)")
    tell = body.index("auto tell")
    after_tell = body.index("};", tell)
    first = body.index("tell(", after_tell)
    assert "map_shared_rank" not in body[:tell] and "map_shared_rank" not in body[after_tell:first]
    before = body[:tell] + body[after_tell:first]
    assert "cluster_barrier()" in before or before.rfind("cluster_wait()") > before.find("cluster_arrive()") >= 0
    # and no CTA leaves while another may still read its shared memory
    assert body.rindex("cluster_barrier()") > body.rindex("tell(")


def test_batch_ctas_that_do_not_run_yet_hold_no_instance():
    """A CTA leaves the batch kernel only when every instance has finished, so
    no instance may wait for a CTA that is not running: instances are taken
    from counters, never by the CTA's index."""
    body = _body(_source("weno_batch.cuh"), "k_batch(BatchArgs b)")
    assert "blockIdx" not in body and "gridDim" not in body
    assert re.search(r"atomicAdd\(&b\.ctrl->prepared", body)


def test_tasks_are_published_after_the_first_lanes_stores():
    """Lane 0 acquires the other CTAs' stores and writes the instance's
    progress, the other lanes of its warp publish tasks too: a barrier that
    orders memory stands between (a shuffle does not)."""
    body = _body(_source("weno_batch.cuh"), "k_batch(BatchArgs b)")
    progress, put = body.index("batch_next_sweep<"), body.index("batch_put(")
    assert "__syncwarp()" in body[progress:put] or "__syncthreads()" in body[progress:put]


def test_a_place_of_the_queue_is_not_filled_while_its_task_is_unread():
    """When the wait for a place runs out, the run ends; the task that nobody
    has read is not overwritten."""
    body = _body(_source("weno_batch.cuh"), "void batch_put(")
    out = body.index("atomicExch(&b.ctrl->abort")
    assert body.index("q->taken") < out < body.index("q->inst = inst")
    assert "return" in body[out:body.index("q->inst = inst")]
