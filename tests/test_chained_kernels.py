"""Kernels launched while the kernel before them still runs (fmm_chain.cuh) may
not promise the compiler that nobody else writes their data: such a kernel is
resident while its predecessor stores what it will read, so a __restrict__
parameter would let loads and stores move before the wait, and const
__restrict__ would allow the non-coherent load path.  Checked on the sources."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_03121_gb300", "csrc")
# the tree's tables, which no kernel writes
TABLES = {"info", "children", "nodes", "leaves", "levels", "levels_df", "off", "rows"}


def _balanced(text, at, pair):
    """End of the bracketed part that opens at text[at]."""
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i + 1
    raise ValueError("unbalanced")


def _kernels():
    """(file, name, parameter list, body) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__\s+void\s*", text):
            at = m.end()
            b = re.compile(r"__launch_bounds__\s*").match(text, at)
            if b:
                at = _balanced(text, b.end(), "()")
            name = re.compile(r"\s*(\w+)\s*").match(text, at)
            end = _balanced(text, name.end(), "()")
            body = re.compile(r"\s*\{").match(text, end)
            if body:
                yield f, name.group(1), text[name.end() + 1:end - 1], text[end:_balanced(text, body.end() - 1, "{}")]


CHAINED = [(f, name, params) for f, name, params, body in _kernels() if "chain_begin()" in body]


def test_the_chained_kernels_are_found():
    names = {name for _, name, _ in CHAINED}
    assert {"p2m_kernel", "m2m_kernel", "m2m_df_kernel", "m2m_df_lanes_kernel", "l2l_kernel", "l2l_leaf_kernel",
            "forces_kernel", "leaf_finish_kernel", "leaf_finish_cells_kernel", "reduce_kernel"} <= names
    # and every kernel that is launched so waits
    launched = set()
    for f in os.listdir(CSRC):
        text = open(os.path.join(CSRC, f)).read()
        launched |= set(re.findall(r"launch_chained\(\s*(\w+_kernel)", text))
    assert launched <= names


@pytest.mark.parametrize("file,name,params", CHAINED, ids=[n for _, n, _ in CHAINED])
def test_only_tables_are_restrict(file, name, params):
    restricted = set(re.findall(r"__restrict__\s+(\w+)", params))
    assert restricted <= TABLES, (file, name, sorted(restricted - TABLES))
