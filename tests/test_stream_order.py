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
    # inline loads through the read-only path: in the two functions that read the register transforms' twiddles
    for m in re.finditer(r"(\w+)\([^()]*\)\s*\{[^{}]*?asm volatile\(\"ld\.global\.nc", text):
        assert m.group(1) in ("tw_load4", "tw_load2"), f"{name}: ld.global.nc in {m.group(1)}"
    assert len(re.findall(r"ld\.global\.nc", text)) == (2 if name == "reg_fft.cuh" else 0), name
    for m in re.finditer(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", text):
        assert m.group(1) in TABLES | {"Gtab", "u"}, f"{name}: const __restrict__ {m.group(1)}"      # Gtab, u: shared memory


@pytest.mark.parametrize("name,text", [pytest.param(n, t, id=n) for n, t in sources() if "launch_dependents" in t])
def test_kernels_wait_before_they_let_their_dependents_start(name, text):
    # What a dependent reads ahead of its own wait (weights, the cached spectrum, tokens) was written in front of the call at the
    # latest.  So no kernel triggers before it has waited, unless it is told that the kernel in front of it has.
    for body in re.split(r"(?=__global__ void|__device__ __forceinline__ void)", text)[1:]:
        first = body.find("launch_dependents")
        if first >= 0:
            before = body[:first]
            assert "after_previous()" in before or "griddepcontrol.wait" in before, f"{name}: {body[:90]}"


def test_level_gates_read_nothing_ahead_of_their_wait():
    # the first kernel of its call: any kernel of the caller's may be in front
    text = dict(sources())["mixer_tc.cu"]
    body = text[text.index("level_gates_kernel(const"):]
    assert not re.search(r"\bW[12]\[|p\.(bw1|bw2|qbar)\[", body[:body.index("after_previous()")])
