"""Kernels that may start before the kernel ahead of them has ended read its results by plain loads.

A non-coherent load is for data that nobody writes while the kernel runs, and may be moved up across
the wait for the kernel ahead; which loads a kernel uses is seen in its source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1602_07483_gb300", "csrc")


def read(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def kernels():
    """name -> source from its __global__ to the next kernel, of every kernel in the headers"""
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cuh"):
            for part in read(f).split("__global__")[1:]:
                out[re.search(r"\b(k_\w+)\(", part).group(1)] = part
    return out


def test_dependent_kernels_use_no_non_coherent_loads():
    src = kernels()
    waits = {n for n, body in src.items() if "pdl_wait()" in body}
    assert {"k_phi_node", "k_phi_moment", "k_uth_pair", "k_uth_moment2"} <= waits
    for n in waits:
        assert not re.search(r"__ldg|ldro\(|\bld<true>|\bld2<true>|pull2<[^>]*true>\(", src[n]), n
        assert src[n].index("pdl_wait()") < re.search(r"ld2?<false>\(|pull2?<", src[n]).start(), n
    # the node-wise loads are written in one place each
    assert "ldro(" not in read("lbpf_nodewise.cuh") + read("lbpf_nodepair.cuh")
    # exactly these kernels are launched so that they may start early
    launched = set(re.findall(r"launch_pdl\((k_\w+)<", read("lbpf_table_impl.cuh")))
    assert launched == waits
