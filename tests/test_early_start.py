"""Kernels that may start while the kernel before them still runs (they call
pdl_wait) must not promise the compiler that what that kernel writes is
constant: a read-only load could be moved above the wait.  Read from the
sources: no GPU."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1507_03392_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))
# what no kernel writes (copies in stream order, which start after and end before every kernel): parameter blocks
# and work list of a batch
CONSTANT_PARAMETERS = {"runs", "items"}
# tables uploaded or rebuilt by copies and by kernels that let nothing start early
CONSTANT_TABLES = ("R.cell", "R.kdt", "R.nanbu", "R.btab", "reinterpret_cast<const uint32_t*>(R.kdt)", "e")


def code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def kernels(text):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(", text):
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params, j, depth = text[m.end():i - 1], text.index("{", i) + 1, 1
        k = j
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        yield m.group(1), params, text[j:k]


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_read_only_parameter_that_a_kernel_writes(path):
    for name, params, body in kernels(code(path)):
        if "pdl_wait()" not in body:
            continue
        const = re.findall(r"const\s+[\w ]+\*\s*__restrict__\s+(\w+)", params)
        assert set(const) <= CONSTANT_PARAMETERS, (name, const)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_loads_stay_below_the_wait(path):
    text = code(path)
    for arg in re.findall(r"__ldg\(((?:[^()]|\([^()]*\))*)\)", text):
        assert re.split(r"\s\+\s", arg)[0] in CONSTANT_TABLES, arg
    assert not re.search(r"asm\s*\(\s*\"ld\.", text)


def test_the_kernels_are_found():
    found = {name for p in SOURCES for name, _, body in kernels(code(p)) if "pdl_wait()" in body}
    assert len(found) == sum(code(p).count("    pdl_wait();") for p in SOURCES) and {"k_one", "k_sort_move"} <= found
