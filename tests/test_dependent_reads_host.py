"""What an earlier launch wrote is not read through the read-only path.

The forward's kernels are launched programmatically dependent (launch_k): one may
be running while its predecessor still writes.  The compiler may move a load through
the read-only path (__ldg, or a `const ... __restrict__` parameter) above the wait
for the predecessor, whatever stands in between, so that path is for the layer's
constants alone.  Shown on the sources: a run that happens to give right results
shows nothing.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2608_07814_gb300", "csrc")
SOURCES = {os.path.basename(p): re.sub(r"//[^\n]*", "", open(p).read())
           for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}
# tables and weights of an installed layer: complete before any forward
CONSTANT_PARAMS = {"paths", "path_len", "rank", "anchors", "corrs", "W", "bias"}
CONSTANT_LOADS = re.compile(r"\b(paths|P\.items|P\.rank|P\.child|P\.kc_child|W|w0|w1)\b")


def _dependent_kernels():
    names = set()
    for src in SOURCES.values():
        for m in re.finditer(r"launch_k\(L,\s*(\w+)", src):
            names.add(m.group(1))
        # a kernel picked by a variable: `auto kern = k_name<...>`
        if re.search(r"launch_k\(L,\s*kern\b", src):
            names.update(re.findall(r"auto kern = (k_\w+)", src))
    names.discard("kern")
    names.discard("void")
    return sorted(n for n in names if n.startswith("k_"))


def _params(name):
    for src in SOURCES.values():
        m = re.search(r"__global__[^;{}]*?\b%s\s*\(" % name, src)
        if m:
            at, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(src[at], 0)
                at += 1
            return src[m.end():at - 1]
    raise AssertionError(name)


def test_the_forward_kernels_are_found():
    found = _dependent_kernels()
    for name in ("k_mark_bits", "k_offsets_plan", "k_assign_rows", "k_bucket_small", "k_router_logits",
                 "k_router_screen", "k_grouped_gemm", "k_swiglu_warp", "k_combine_tok", "k_tc_gemm",
                 "k_stream_gemm", "k_ct_swiglu"):
        assert name in found


@pytest.mark.parametrize("name", _dependent_kernels())
def test_read_only_parameters_are_layer_constants(name):
    for p in _params(name).split(","):
        if "__restrict__" in p and re.search(r"\bconst\b[^*]*\*", p):
            assert p.split()[-1] in CONSTANT_PARAMS, p.strip()


def test_read_only_loads_are_of_layer_constants():
    for f, src in SOURCES.items():
        if "launch_k(" not in src:
            continue
        for m in re.finditer(r"__ldg\(", src):
            arg = src[m.end():src.index(";", m.end())]
            assert CONSTANT_LOADS.search(arg), (f, arg)
