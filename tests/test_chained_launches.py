"""Programmatic launches, from the sources alone: a kernel that may start while
its predecessor is still running does nothing before it has waited for it."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1010_3816_gb300", "csrc")


def _sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            text = open(os.path.join(CSRC, name)).read()
            yield name, re.sub(r"//[^\n]*", "", text)


def test_only_chain_start_orders_chained_kernels():
    """The two instructions stand in chain_start alone, the wait right after the
    release of the next launch."""
    found = [(name, m) for name, text in _sources() for m in re.findall(r"griddepcontrol\.(\w+)", text)]
    assert found == [("tk_stencil.cuh", "launch_dependents"), ("tk_stencil.cuh", "wait")]


def test_chained_kernels_wait_first():
    """Every kernel handed to launch_chained calls chain_start before any other
    statement (constants and the declarations of shared memory aside)."""
    kernels, calls = {}, set()
    for _, text in _sources():
        for m in re.finditer(r"__global__[^{;]*?\b(\w+_kernel)\s*\([^{;]*\)\s*\{", text):
            kernels[m.group(1)] = text[m.end():]
        for m in re.finditer(r"\b(?:launch_chained<|TK_CHAINED\(\()(\w+)", text):
            calls.add(m.group(1))
    chained = {c for c in calls if c.endswith("_kernel")}
    assert len(chained) >= 4
    for name in chained:
        for line in kernels[name].split(";"):
            line = line.strip()
            if re.match(r"(if \(kUsePDL\) )?chain_start\(\)$", line):
                break
            assert re.match(r"(constexpr|(extern )?__shared__)\b", line), (name, line)


def test_programmatic_edge_only_for_kernels_without_a_stack_frame():
    """The launch attribute stands in launch_chained alone, and goes with the launch
    only where the kernel has no local memory."""
    where = [(name, text) for name, text in _sources() if "ProgrammaticStreamSerialization" in text]
    assert [name for name, _ in where] == ["tk_stencil.cuh"]
    text = where[0][1]
    assert text.count("cudaLaunchAttributeProgrammaticStreamSerialization") == 1
    body = text[text.index("cudaError_t launch_chained("):]
    body = body[:body.index("cudaLaunchKernelEx")]
    assert re.search(r"bool chained = frameless\(\(const void \*\)kern\);", body)
    assert re.search(r"numAttrs = chained \? 1 : 0;", body)
    assert re.search(r"frameless\(const void \*kern\)\s*\{[^}]*localSizeBytes == 0", text)
