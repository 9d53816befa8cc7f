"""Kernels launched as programmatic dependents may be resident before the kernel ahead of them
has written its results, and see them only after their wait.  The read-only path (__ldg, or a
const pointer marked __restrict__) promises data that is constant while the kernel is resident
and may be read at any point of it, so such kernels use it for biases and output weights only, which
were written at least two kernels earlier."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_15183_gb300", "csrc")


def _code(name):
    src = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", src)


def _block(src, i):
    """The text from the first '{' at or after i to its closing brace."""
    i = src.index("{", i)
    depth = 0
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if not depth:
            return src[i:j + 1]
    raise ValueError("unbalanced")


def _dependents():
    found = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cu"):
            src = _code(name)
            for m in re.finditer(r"__global__ void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(([^{;]*)\)\s*{", src):
                body = _block(src, m.end() - 1)
                wait = re.search(r"\b(?:pdl_wait|after_wait)\(\)", body)
                if wait:
                    found.append((name, m.group(1), m.group(2), body[wait.end():]))
    return found


def test_the_scan_finds_the_dependent_kernels():
    names = {k for _, k, _, _ in _dependents()}
    assert {"fused_single", "fused_batch", "fill_only", "fill_keys", "imb_band", "conv3x3_rows", "conv3x3_halo",
            "conv3x3_tc", "conv3x3_dw", "dw_reduce_kernel", "dz_kernel", "out_bwd_kernel", "weights_kernel"} <= names


@pytest.mark.parametrize("name,kernel,params,after", [pytest.param(*d, id=f"{d[0]}:{d[1]}") for d in _dependents()])
def test_no_read_only_loads_after_the_wait(name, kernel, params, after):
    assert not re.search(r"\bconst\b[^,]*__restrict__", params), f"{kernel}: {params}"
    assert not re.search(r"__ldg\((?!a\.(bias|wout)\b)", after)
    if name == "fused.cu":  # its device functions run after the waits too
        assert "__ldg(" not in _code(name)
