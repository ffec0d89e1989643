"""Memory ordering of the cluster kernels' barriers, read from the sources.

A cluster barrier whose arrival is relaxed orders nothing that came before it
(PTX ISA, barrier.cluster): what other blocks read or write across it needs a
fence at cluster scope first, by a thread that the block's other threads have
reached at a block barrier."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_relaxed_arrivals_follow_a_cluster_fence():
    for path in glob.glob(os.path.join(ROOT, "paper_2309_09064_gb300", "csrc", "*.cu*")):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"barrier\.cluster\.arrive\.relaxed", code):
            before = code[:m.start()]
            block = before.rfind("__syncthreads()")
            fence = before.rfind("fence.acq_rel.cluster")
            wait = before.rfind("barrier.cluster.wait")
            assert max(wait, -1) < block < fence, f"{os.path.basename(path)}: relaxed arrival without a release"
