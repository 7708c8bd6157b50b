"""Kernels that may start under their predecessor (launch_pdl) read what it wrote: plain loads only.  The non-coherent path
(`__ldg`, `const T* __restrict__` parameters) is for memory that nobody writes while the kernel lives, and such a load may be
moved in front of the wait for the predecessor."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_20971_b200", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def _kernels(code):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\(([^{;]*?)\)\s*\{", code):
        depth, at = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(code[at], 0)
            at += 1
        yield m.group(1), m.group(2), code[m.end():at]


def test_every_dependent_launch_is_of_a_kernel_that_waits():
    waiting = {n for f in SOURCES for n, _, body in _kernels(_code(f)) if "pdl_wait()" in body}
    assert {"plan_rows_kernel", "combine_parts_kernel", "prefill_duo_kernel", "select_prep_kernel", "select_pair_kernel",
            "select_tc_kernel", "density_kernel", "block_stats_warp_kernel"} <= waiting
    for f in SOURCES:
        for name in re.findall(r"launch_pdl\((\w+_kernel)", _code(f)):
            assert name in waiting


@pytest.mark.parametrize("source", SOURCES)
def test_no_load_of_a_dependent_kernel_is_non_coherent(source):
    code = _code(source)
    for name, params, body in _kernels(code):
        if "pdl_wait()" in body:
            assert not re.search(r"\bconst\b[^,]*__restrict__", params), name
    # helpers of those kernels; next_block serves prefill_mma_kernel, which starts when everything before it has ended
    helpers = re.sub(r"int next_block\(.*?\n\}", "", code, flags=re.S)
    assert "__ldg" not in helpers
