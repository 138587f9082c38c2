"""What the kernels' sources promise the compiler about memory that other kernels write (read on the CPU: the kernels of a chain
are resident while their predecessors write)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_18394_b200", "csrc")
TABLES = {"tab", "tw", "Fg", "Ag", "p.twq", "p.twr"}           # built by spectre_create, never written again


def sources():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(f).read())
        yield os.path.basename(f), text


@pytest.mark.parametrize("name,text", [pytest.param(n, t, id=n) for n, t in sources()])
def test_read_only_loads_and_restrict_are_for_the_contexts_tables(name, text):
    for m in re.finditer(r"__ldg\(\s*([\w.]+)", text):
        assert m.group(1) in TABLES, f"{name}: __ldg of {m.group(1)}"
    for m in re.finditer(r"__global__ void(?:\s+__launch_bounds__\((?:[^()]|\([^()]*\))*\))?\s+(\w+)\(([^{;]*)\)\s*\{", text):
        if not re.match(r"(build_|reg_table)", m.group(1)):
            assert "__restrict__" not in m.group(2), f"{name}: {m.group(1)}"
    for m in re.finditer(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", text):
        assert m.group(1) in TABLES | {"Gtab", "u"}, f"{name}: const __restrict__ {m.group(1)}"      # Gtab, u: shared memory
