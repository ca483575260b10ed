"""A kernel that runs CTA-pair instructions declares its cluster of two itself.  As a launch
attribute alone it can be lost (a profiler relaunching a cooperative kernel drops it), and the
pair instructions then run outside a cluster."""
import glob
import os
import re

from conftest import ROOT


def test_pair_kernels_declare_their_cluster():
    found = set()
    for path in glob.glob(os.path.join(ROOT, "paper_2607_03011_gb300", "csrc", "*.cu")):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        kernels = list(re.finditer(r"__global__\s+void\s+([^;{]*?)(\bk_\w+)\s*\([^;{]*\{", src))
        for k, nxt in zip(kernels, kernels[1:] + [None]):
            body = src[k.end():nxt.start() if nxt else len(src)]
            if "tmem_alloc_pair(" in body:
                found.add(k[2])
                assert "__cluster_dims__(2, 1, 1)" in k[1], k[2]
    assert found == {"k_gemm_split", "k_polar_loop"}
