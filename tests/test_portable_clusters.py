"""Kernels launched in clusters run wherever the library loads: clusters of more than 8 CTAs (the portable
size) only after the device has said that it has room for one, with a portable size to fall back to.
A partitioned GPU may have no GPC with 16 SMs to give."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1801_09803_gb300", "csrc")


def test_large_clusters_have_a_portable_fallback():
    seen = 0
    for f in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, f)).read()
        src = re.sub(r"//[^\n]*", "", src)
        if "cudaFuncAttributeNonPortableClusterSizeAllowed" in src:
            seen += 1
            assert "cudaOccupancyMaxActiveClusters" in src, f
        for m in re.finditer(r"constexpr int (PF_CL\w*) = (\d+)", src):
            assert int(m.group(2)) <= 8 or m.group(1) == "PF_CL_LARGE"
    assert seen <= 1
