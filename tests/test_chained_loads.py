"""The read-only path in kernels launched as a programmatic chain. Such a kernel is resident before its
predecessors have written, and __ldg and const __restrict__ promise data that does not change while
the kernel runs: only a plan's constant tables may be read that way (the sources are read as text)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_12616_gb300", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))
# instance table, block prefixes, block and tile tables, cosines of the coefficient nodes
CONSTANT = {"insts", "pre", "tab", "w.tab", "ct"}


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def functions(text):
    """(head, body) of every __global__ and __device__ function."""
    for m in re.finditer(r"__(?:global|device)__\b[^;{}]*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(0), text[m.end():i]


@pytest.mark.parametrize("name", FILES)
def test_ldg_reads_constant_tables_only(name):
    for arg in re.findall(r"__ldg\(\s*([A-Za-z_][\w.]*)", code(name)):
        assert arg in CONSTANT, f"{name}: __ldg({arg} ...)"


@pytest.mark.parametrize("name", FILES)
def test_restrict_parameters_of_chained_kernels(name):
    text = code(name)
    seen = 0
    for head, body in functions(text):
        kernel = "__global__" in head
        if kernel and not re.search(r"\bpdl_(?:sync|wait)\(\)", body):
            continue   # launched plainly
        seen += kernel
        for param in re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", head):
            assert param in CONSTANT, f"{name}: {param} in {head.split('(')[0].split()[-1]}"
    if name in ("coef.cu", "gemm_digits.cu", "gemm_tc.cu", "lanczos.cu", "reduce.cu"):
        assert seen > 0


def test_every_chained_launch_waits():
    """Each kernel named in a launch_pdl call waits in its body (k_tc_gemm: in its unchained form)."""
    bodies = {}
    for name in FILES:
        for head, body in functions(code(name)):
            m = re.findall(r"\b(k_\w+)\s*\(", head)
            if "__global__" in head and m:
                bodies[m[-1]] = body
    for name in FILES:
        for kern in re.findall(r"launch_pdl\(\s*(?:[\w.]+\s*,\s*)?(k_\w+)", code(name)):
            assert re.search(r"\bpdl_(?:sync|wait)\(\)", bodies[kern]), kern
