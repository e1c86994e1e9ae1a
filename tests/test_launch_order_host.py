"""Every kernel that is launched while the one before it drains waits for it before its
first access to global memory.  Read-only loads (__ldg, pointers declared __restrict__)
may be moved above that wait unless their address depends on its result, so a file that
has them may not drop the result.  Read from the sources: no GPU, no build."""
import os
import re

import pytest

from paper_2608_23463_gb300.buildlib import CSRC

FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
READ_ONLY = re.compile(r"__ldg\(|__restrict__|ld\.global\.nc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _kernels(code):
    """(name, body) of each __global__ function defined in code."""
    for m in re.finditer(r"__global__", code):
        brace = code.index("{", m.end())
        name = re.findall(r"(\w+)\s*\(", code[m.end():brace].replace("__launch_bounds__(", " "))
        name = [n for n in name if not n.startswith("__")][0]
        depth, i = 1, brace + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            i += 1
        yield name, code[brace:i]


@pytest.mark.parametrize("name", FILES)
def test_kernels_wait_and_reads_depend_on_it(name):
    code = _code(name)
    for kernel, body in _kernels(code):
        if kernel == "ffma_probe_kernel":  # an ordinary launch: it waits by itself
            continue
        calls = re.findall(r"([^;{}]*)\bpdl_enter\(\)", body)
        assert len(calls) == 1, f"{kernel}: {len(calls)} waits"
        if READ_ONLY.search(code):
            var = re.fullmatch(r"\s*const int (\w+) = (?:\w+ \+ )?", calls[0])
            assert var, f"{kernel} drops the wait's result beside read-only loads"
            assert len(re.findall(rf"\b{var[1]}\b", body)) > 1, f"{kernel}: {var[1]} is unused"
