"""Rules of the kernels' synchronisation that a missed case would break only
now and then on the GPU, checked on the source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_16843_gb300", "csrc")


def kernels(name):
    """{kernel: body} of one source file, comments removed."""
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    out = {}
    for m in re.finditer(r"__global__ void[^{;]*?\b(k_\w+)\(", text):
        start = text.index("{", m.end())
        depth, end = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
            if depth == 0:
                break
        out[m[1]] = text[start:end]
    return out


def test_cluster_kernels_start_together():
    """A store to another CTA's shared memory is defined only once that CTA has
    started: every kernel that runs on a cluster passes a cluster barrier
    before its first such store and before it enters the step code, whose
    first operation may be a reduction."""
    found = {k: b for k, b in kernels("k_persist.cu").items() if "ClusterX x{" in b}
    assert set(found) == {"k_step_cluster", "k_batch_cluster"}
    for name, body in found.items():
        barrier = body.index("ClusterX::cluster_barrier()") if "ClusterX::cluster_barrier()" in body else len(body)
        first = min(i for i in (body.find("run_steps<"), body.find("st_cluster(")) if i >= 0)
        assert barrier < first, name
