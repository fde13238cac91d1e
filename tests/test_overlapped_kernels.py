"""Kernels that may be resident while the kernel before them still writes what
they read (every kernel that calls pdl_wait): their sources promise no
read-only data (`__restrict__` parameters, `__ldg`, `ld.global.nc`), and every
kernel that is launched that way does wait."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2603_20966_gb300", "csrc")


def _sources():
    text = {}
    for f in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(f) as fh:
            text[os.path.basename(f)] = re.sub(r"//[^\n]*", "", fh.read())
    return text


def _kernels(text):
    """name -> (parameter list, body) of every __global__ function."""
    out = {}
    for src in text.values():
        for m in re.finditer(r"__global__\s+void(?:\s+__launch_bounds__\([^)]*\))?\s+(k_\w+)\s*\(",
                             src):
            i, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            params = src[m.end():i - 1]
            j = src.index("{", i)
            e, depth = j + 1, 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[e], 0)
                e += 1
            out[m.group(1)] = (params, src[j:e])
    return out


def test_overlapped_kernels_wait_and_read_with_ordinary_loads():
    text = _sources()
    kernels = _kernels(text)
    launched = set()
    for src in text.values():
        for m in re.finditer(r"launch_overlapped\(([^;]*);", src):
            launched |= set(re.findall(r"\bk_\w+", m.group(1)))
    assert {"k_splitk_reduce", "k_splitk_reduce_batched", "k_reduce_segments",
            "k_sketch_fp32_left", "k_sketch_bf16x2_left", "k_sketch_bf16x2_right",
            "k_sketch_e4m3_right"} <= launched
    for name in launched:
        assert "pdl_wait()" in kernels[name][1], name
    for name, (params, body) in kernels.items():
        if "pdl_wait()" in body:
            assert "__restrict__" not in params, name
            assert "__ldg" not in body and "ld.global.nc" not in body, name
    # the sums that the reductions share
    assert "__restrict__" not in text["sk_reduce.cuh"]
