"""Programmatic dependent launch: a kernel so launched is alive while the one
before it still writes, so what it reads of that must stay behind its wait.

Read from the sources (no GPU): every such kernel waits; none of its inputs but
the plan's tables is a const __restrict__ parameter (which the compiler may read
through the read-only path, whose data must not change while the kernel is
alive) or read by __ldg; and no assembly load is movable or read-only."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1208_3210_gb300", "csrc")
FILES = {os.path.basename(f): re.sub(r"//[^\n]*", "", open(f).read())
         for f in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))}
# laid out when the plan is made: constant while any kernel of a call is alive
TABLES = {"tab", "tw", "ptw", "etw"}
# what __ldg may read: the tables, and the names by which helpers know their rows
ROWS = TABLES | {"row", "wt", "w4", "src"}
DEPENDENT = sorted(f for f, s in FILES.items() if f.endswith(".cu") and "launch_after(" in s)


def _kernels(text):
    """(name, parameters, text up to the next kernel)."""
    found = list(re.finditer(r"__global__[^{;]*?\b(k_\w+)\s*\(([^{;]*?)\)\s*\{", text, re.S))
    for m, n in zip(found, found[1:] + [None]):
        yield m.group(1), " ".join(m.group(2).split()), text[m.end():n.start() if n else len(text)]


def test_files_found():
    assert len(DEPENDENT) >= 10


@pytest.mark.parametrize("name", DEPENDENT)
def test_kernels_wait_and_read_with_ordinary_loads(name):
    text = FILES[name]
    plain = set(re.findall(r"\b(k_\w+)(?:<[^;{}<>]*>)?\s*<<<", text))
    for kernel, params, body in _kernels(text):
        if kernel in plain:
            continue
        assert "after_previous();" in body, f"{kernel} does not wait"
        for p in params.split(","):
            if "const" in p and "__restrict__" in p:
                assert p.split()[-1] in TABLES, f"{kernel}: {p.strip()}"


@pytest.mark.parametrize("name", sorted(FILES))
def test_loads_stay_behind_the_wait(name):
    text = FILES[name]
    assert "ld.global.nc" not in text
    for m in re.finditer(r"asm\s*(volatile)?\s*\(\s*\"([^\"]*)", text):
        assert m.group(1) or "ld.global" not in m.group(2), m.group(0)
    if name.endswith(".cuh") or name in DEPENDENT:
        for arg in re.findall(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\()?\s*&?(\w+)", text):
            assert arg in ROWS, f"__ldg({arg}...)"
