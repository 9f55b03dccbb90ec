"""Static checks of the CUDA sources (no GPU): which kernels may reach into the
shared memory of other blocks, and that they look at their cluster first."""
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


def test_kernels_with_peers_check_their_cluster():
    """Every kernel that calls pencil_split (stores to peers) compares the
    cluster it runs in with the one it was launched for before that call."""
    seen = 0
    for f in sorted(os.listdir(CSRC)):
        for k in re.split(r"__global__", _code(f))[1:]:
            at = k.find("pencil_split<")
            if at < 0:
                continue
            seen += 1
            check = re.search(r"if \(cluster_size\(\) != C \|\| c != \(int\)\(blockIdx\.x % C\)\)", k[:at])
            assert check and "return;" in k[check.end():at], f
    assert seen == 1
