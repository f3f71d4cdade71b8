"""Kernels that may start before the launch before them has ended (they call pdl_wait) read what that
launch writes by plain loads: no __ldg, and no const __restrict__ pointer to the values of Eq. 1 that
x0_values_kernel leaves for the gathers."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1801_10016_gb300", "csrc")


def kernels():
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        text = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"__global__ void (?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(([^{;]*)\) \{", text):
            end = text.index("\n}\n", m.end())
            yield m.group(1), m.group(2), text[m.end():end]


def test_dependent_launches_read_by_plain_loads():
    seen = set()
    for name, params, body in kernels():
        if "pdl_wait();" not in body:
            continue
        seen.add(name)
        assert "__ldg(" not in body, name
        assert not re.search(r"const double\* __restrict__ x0\b", params), name
    assert {"bounds_kernel", "gather_kernel", "oz_gather_kernel", "gather_lp_kernel", "oz_step_kernel",
            "square_tc_persistent_kernel", "x0_values_kernel"} <= seen
    helper = open(os.path.join(CSRC, "gsp2_internal.cuh")).read()
    params = re.search(r"void gather_column\(([^{]*)\) \{", helper).group(1)
    assert "const double* xq" in params
