"""Kernels that start before their predecessor ends may prefetch only what no kernel
writes meanwhile.  A `const T *__restrict__` parameter lets the compiler load through
the read-only path and move the load above griddepcontrol.wait, so in the solve phase
the qualifier stands only on data that setup leaves fixed."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1403_1649_gb300", "csrc")

# matrix entries, aggregates, interpolation and smoother weights, system offsets and maps
FIXED = {"agg", "amem", "aptr", "pw", "pwm", "pw64", "wd", "wdc", "Ainv", "binv", "boff", "off", "sys", "sysc",
         "sptr", "scol", "sval", "spair", "sdiag"}


def kernels(source):
    """name, parameter list and body of every kernel."""
    for m in re.finditer(r"__global__[^{;]*?\b(k_\w+)\s*\(([^{]*?)\)\s*\{", source, re.S):
        depth, end = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(source[end], 0)
            end += 1
        yield m.group(1), m.group(2), source[m.end():end]


@pytest.mark.parametrize("name", ["solve.cu", "tail.cu"])
def test_restrict_only_on_fixed_data(name):
    with open(os.path.join(CSRC, name)) as f:
        source = f.read()
    seen, wrong = 0, []
    for kernel, params, body in kernels(source):
        if "pdl_wait" not in body:
            continue
        seen += 1
        for p in re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", params):
            if p not in FIXED:
                wrong.append(f"{kernel}: {p}")
    assert seen and not wrong, wrong
