"""Static checks of the CUDA sources (no GPU): which kernels may reach into the
shared memory of other blocks."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2202_12477_gb300", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def test_cooperative_kernels_launch_without_clusters():
    """A cooperative launch here has no cluster and no store to another block's
    shared memory: the combination faulted on the GPU under a profiler."""
    seen = 0
    for f in sorted(os.listdir(CSRC)):
        text = _code(f)
        if "Cooperative" not in text:
            continue
        seen += 1
        assert not re.search(r"ClusterDimension|mapa|\bpeer\(|barrier\.cluster|cluster_(arrive|wait)|pencil_split", text), f
    assert seen
