"""Properties of the kernels' sources that no run shows as long as the compiler is kind."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0912_3912_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_aligned_cluster_barrier_after_the_warp_has_met():
    body = re.search(r"void cluster_sync\(\) \{(.*?)\n\}", _source("tc.cuh"), re.S).group(1)
    assert body.index("__syncwarp();") < body.index("barrier.cluster.arrive.release.aligned")
    for name in sorted(os.listdir(CSRC)):  # ... and no such barrier elsewhere
        assert name == "tc.cuh" or "barrier.cluster" not in _source(name), name


def test_dynamic_shared_memory_is_declared_aligned():
    """Kernels read it in 16-byte vectors; its base follows the static variables.  (Two
    kernels round the address up to 1,024 bytes themselves.)"""
    found = 0
    for name in sorted(os.listdir(CSRC)):
        src = _source(name)
        for m in re.finditer(r"extern __shared__ ([^;]*);", src):
            found += 1
            assert "__align__(16)" in m.group(1) or "1023" in src[m.end(): m.end() + 400], (name, m.group(0))
    assert found >= 8
