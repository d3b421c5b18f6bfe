"""Rules of the kernel sources that no result shows: broken, they cost speed or
rely on what the hardware does not promise.  Read from the sources, on the CPU."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_1611_02045_gb300" / "csrc"


def source(name):
    """The file without its // comments."""
    return re.sub(r"//[^\n]*", "", (CSRC / name).read_text())


def test_cluster_kernels_read_their_arguments_in_place():
    """A by-value argument struct is copied, and its size then steers the register
    allocation of kernels whose text did not change."""
    heads = re.findall(r"__global__[^{;]*?\b(cluster_apply_H\w*)\(([^)]*)\)", source("gpe_cluster.cuh"))
    assert {name for name, _ in heads} == {"cluster_apply_H", "cluster_apply_H_stream"}
    for name, args in heads:
        assert re.fullmatch(r"const __grid_constant__ ClusterHArgs \w+", args.strip()), (name, args)
