"""Kernels launched programmatically may run while the kernel in front of them still
writes: they must not read through the non-coherent path, which needs the data
unchanged for the kernel's whole life.  Checked on the source of the network's kernels."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_05943_gb300", "csrc")


def _function(src, name):
    """Parameter list and body of the (first) definition of a function."""
    i = re.search(r"\bvoid (?:__launch_bounds__\([^)]*\) )?(?:\n\s+)?" + name + r"\(|\b" + name + r"\(const __grid_constant__", src).start()
    j = src.index("{", i)
    depth, k = 0, j
    while True:
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        k += 1
        if depth == 0:
            return src[i:j], src[j:k]


def test_dependent_kernels_read_coherently():
    src = open(os.path.join(CSRC, "nop_kernels.cu")).read()
    names = set(re.findall(r"launch_pdl\((k_\w+)", src)) | {"k_conv_tma", "k_conv_row"}   # the last two by a variable
    assert {"k_wgrad_row", "k_dgrad_small", "k_pool2_bwd_skip8"} <= names
    helpers = {n for n in re.findall(r"__device__ __forceinline__ void (tm_\w+)\(", src)}
    for name in names | helpers:
        params, body = _function(src, name)
        assert not re.search(r"const [\w]+\* __restrict__", params), name
        assert "__ldg" not in body and ".global.nc" not in body, name
