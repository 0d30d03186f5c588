"""Distributed shared memory may be touched only once the other CTAs of the cluster are known to run: in every kernel of
the readout the first access to another CTA's shared memory comes after a cluster barrier that all of its CTAs have
arrived at. A missing one shows on no run (the loads before it hide it), so the source is read."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2201_05529_gb300", "csrc")


def _kernels(src):
    for m in re.finditer(r"__global__[^;{]*?(k_\w+)\(", src):
        at = src.index("{", m.end())
        depth, end = 1, at + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[end], 0)
            end += 1
        yield m.group(1), src[at:end]


def test_remote_shared_memory_after_a_cluster_barrier():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "readout.cu")).read())
    seen = 0
    for name, body in _kernels(src):
        remote = body.find("map_shared_rank")
        if remote < 0:
            continue
        seen += 1
        done = [i for i in (body.find("cl.sync()"), body.find("barrier_wait(")) if i >= 0]
        assert done and min(done) < remote, name
    assert seen == 2
