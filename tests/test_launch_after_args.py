"""Kernels that may start while the one before them runs (launch_after): the arrays which that one writes are not
`__restrict__` parameters, which would allow the compiler to load them before the wait."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1612_00474_gb300", "csrc")
# written by earlier kernels that have ended before such a kernel can start, by the host, or by the kernel itself
SETTLED = {"row_seg", "col_start", "col_rows", "tile_inst", "active", "sinst", "F", "T", "P", "U", "U2"}


def test_early_kernels_take_plain_pointers():
    text = "".join(open(f).read() for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))))
    kernels = set(re.findall(r"launch_after\(\s*[^;]*?,\s*(\w+_kernel)\b", text))
    assert kernels == {"pair_sym_reduce_kernel", "pair_sym64_reduce_kernel", "gs_cluster_kernel"}
    for k in kernels:
        args = re.search(r"__global__[^;{]*?\b" + k + r"\(\s*([^{]*?)\)\s*\{", text).group(1)
        restricted = set(re.findall(r"__restrict__\s+(\w+)", args))
        assert restricted <= SETTLED, (k, restricted - SETTLED)
