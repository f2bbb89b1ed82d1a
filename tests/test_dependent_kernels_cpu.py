"""Kernels launched as programmatic dependents are resident while the kernel before them still writes
what they read after the wait.  Their sources may not load it as read-only data: a const __restrict__
parameter or __ldg becomes a non-coherent load, which promises nothing about such writes."""
import glob
import os
import re

import pytest

import paper_cs_9809105_gb300 as h

CSRC = os.path.join(os.path.dirname(h.__file__), "csrc")
CODE = re.compile(r"//[^\n]*|/\*.*?\*/", re.S)


def kernels(text):
    """(name, parameters, body) of every kernel of a source without comments."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^;{]*?\)\s+)?(\w+)\s*\(", text):
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params = text[m.end():i - 1]
        j = k = text.index("{", i)
        depth = 1
        while depth:
            k += 1
            depth += {"{": 1, "}": -1}.get(text[k], 0)
        yield m.group(1), params, text[j:k]


SOURCES = {os.path.basename(p): CODE.sub("", open(p).read()) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}
WAITING = [(f, n, p) for f, t in SOURCES.items() for n, p, b in kernels(t) if "pdl_wait()" in b]


def test_the_scan_finds_the_kernels():
    names = {n for _, n, _ in WAITING}
    assert {"gemv_reduce", "gemv_f32_n_vec", "gemv_t_vec", "gemm_f64_kernel", "gemm_z64_kernel", "nbody_tiled",
            "ozaki_split_w_kernel", "ozaki_recombine_kernel", "gemm_ozaki_pair_kernel", "gemm_tc_pair_kernel",
            "gemm_tc_split_kernel", "gemm_grouped_pair_kernel"} <= names


@pytest.mark.parametrize("source,name,params", WAITING, ids=lambda v: v if re.fullmatch(r"[\w.]+", v) else "")
def test_no_read_only_parameters(source, name, params):
    assert not [p for p in params.split(",") if "__restrict__" in p and "const" in p], (source, name)


@pytest.mark.parametrize("source", sorted({f for f, _, _ in WAITING}))
def test_no_read_only_loads(source):
    assert not re.search(r"\b__ldg\b|\.nc\.", SOURCES[source]), source
