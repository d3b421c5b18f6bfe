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


def kernels(text):
    """(name, parameters, body) of each __global__ function."""
    for m in re.finditer(r"__global__[^{;]*?\b(\w+)\(([^)]*)\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m[1], m[2], text[m.end() : i]


def test_kernels_launched_early_read_fields_coherently():
    """A kernel that may start while the one in front of it still writes must not read
    through the non-coherent path (__ldg, const __restrict__) what that one may write.
    V and the tables of a context are written by no kernel of a chain."""
    seen = 0
    for name in ("gpe_adjoint.cu", "gpe_misc.cu"):
        for kernel, params, body in kernels(source(name)):
            if "pdl_wait()" not in body:
                continue
            seen += 1
            assert "__ldg(" not in body, (name, kernel)
            for p in params.split(","):
                if "__restrict__" in p and p.strip().startswith("const"):
                    assert re.search(r"__restrict__ V$", p.strip()), (name, kernel, p)
    assert seen >= 9
