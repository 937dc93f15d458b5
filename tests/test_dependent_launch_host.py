"""Kernels launched as programmatic dependents read no memory through the read-only path (CPU only).

Such a kernel starts while the kernel before it on the stream may still be writing. Its own order
is kept by wait_previous(), but __ldg, ld.global.nc and the loads that the compiler may make of a
``const T* __restrict__`` parameter are defined only for memory that nobody writes during the
kernel's whole life, and may move above the wait. These checks read the sources: every kernel
that launch_dep starts, and every function of the sources that it calls.
"""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2501_03759_gb300", "csrc")
FILES = ("lbch_api.cu", "lbch_aux.cuh", "lbch_batch.cuh", "lbch_lattice.cuh", "lbch_step.cuh", "lbch3.cuh", "lbch_f2.cuh")
NOT_FUNCTIONS = {"if", "for", "while", "switch", "catch", "return", "sizeof", "defined", "constexpr"}
# Tables that are uploaded and waited for before the first launch that reads them.
CONSTANT_TABLES = {"Field", "int4"}


def sources():
    text = ""
    for name in FILES:
        with open(os.path.join(CSRC, name)) as fh:
            text += re.sub(r"//[^\n]*|/\*.*?\*/", "", fh.read(), flags=re.S) + "\n"
    return text


def balanced(text, at, pair):
    depth = 0
    for k in range(at, len(text)):
        depth += (text[k] == pair[0]) - (text[k] == pair[1])
        if depth == 0:
            return k + 1
    raise AssertionError("unbalanced source")


def functions(text):
    """name -> [(parameters, body)] of every function the sources define (overloads together)."""
    found = {}
    for m in re.finditer(r"\b(\w+)\s*\(", text):
        if m.group(1) in NOT_FUNCTIONS:
            continue
        end = balanced(text, m.end() - 1, "()")
        tail = re.match(r"\s*(?:const\s*)?\{", text[end:])
        if tail:
            body_at = end + tail.end() - 1
            found.setdefault(m.group(1), []).append((text[m.end():end - 1], text[body_at:balanced(text, body_at, "{}")]))
    return found


TEXT = sources()
FUNCTIONS = functions(TEXT)
KERNELS = sorted(set(re.findall(r"launch_dep\(\s*(?:lbch3::)?(\w+_kernel)\b", TEXT)))


def reached(name):
    seen, todo = set(), [name]
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        for _, body in FUNCTIONS[f]:
            todo += [g for g in re.findall(r"\b(\w+)\b", body) if g in FUNCTIONS]
    return seen


def test_the_dependent_kernels_are_found():
    assert {"step_kernel", "step_batch_kernel", "phi_kernel", "mass_kernel", "energy_kernel", "final_sum_kernel",
            "gather3_kernel", "mu3_kernel", "stream3_kernel"} <= set(KERNELS)
    assert all(k in FUNCTIONS for k in KERNELS)
    assert "issue_row" in reached("step_kernel")


@pytest.mark.parametrize("kernel", KERNELS)
def test_dependent_kernel_waits_and_reads_no_read_only_path(kernel):
    calls = reached(kernel)
    assert "wait_previous" in calls
    for f in sorted(calls):
        for params, body in FUNCTIONS[f]:
            assert "__ldg" not in body and not re.search(r"ld\.global[\w.:]*\.nc", body), f
            for t in re.findall(r"const\s+([\w:]+)\s*\*\s*__restrict__", params):
                assert t in CONSTANT_TABLES, (f, t)
            # an inline load is tied to the wait before it
            for asm, text in re.findall(r"\basm(\s+volatile)?\s*\(([^;]*ld\.global[^;]*)\)\s*;", body):
                assert asm and '"memory"' in text, f
