"""Rules that the kernels' sources keep and that no run can show.

Kernels of a step live while the one before them still writes the fields, so only tables and factors, which nothing
writes then, may be read through the read-only path.  __syncthreads stands in no branch that the warps of a CTA take
differently.
"""
import os
import re

from paper_2604_19370_gb300 import build


def _code(name):
    with open(os.path.join(build.CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_read_only_loads_are_of_tables():
    # what the line passes read so: parts of a factor table (p, U, T of add_state, tab), rows of the explicit operator
    allowed = re.compile(r"__ldg\((reinterpret_cast<const (float|double)[24]\*>\(p|p\)|U \+|T \+ a \* PD|static_cast<const int\*>\("
                         r"(tab|shift\(tab)|band \+)")
    for name in sorted(os.listdir(build.CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            code = _code(name)
            assert len(re.findall(r"__ldg\(", code)) == len(allowed.findall(code)), name
            if name != "wf_lines.cuh":
                assert "__ldg" not in code, name


def test_no_cta_barrier_in_a_warps_own_branch():
    code = _code("wf_quad.cuh")
    code = code[code.index("void quad_rows("):]
    at = code.index("if (__builtin_expect(hot, 0)) {")  # the rows of a warp reach a fire
    depth, end = 0, at
    while True:  # to the end of the branch and of its else
        depth += {"{": 1, "}": -1}.get(code[end], 0)
        end += 1
        if depth == 0 and code[end - 1] == "}" and not code[end:].lstrip().startswith("else"):
            break
    assert "__syncthreads" not in code[at:end] and "cta_barrier" in code[at:end]
