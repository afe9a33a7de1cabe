"""Kernels of a programmatic launch chain take their tensor memory before they let dependents start.

A dependent CTA may start once every CTA of the grid before it has called pdl_begin, and it allocates
its own tensor memory before it waits for that grid. A CTA that called pdl_begin first and then had to
wait for columns held by a dependent would close a circle of waits. The order is a property of the
source: in every kernel that does both, the allocation comes first and the warp that made it calls
pdl_begin (or a block barrier lies between them).
"""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_14025_gb300", "csrc")


def kernels():
    """(file, name, body) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__", src):
            name = re.search(r"\b(k_\w+)\s*\(", src[m.start():])
            i = src.index("{", m.start() + name.end())
            depth, j = 1, i + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(src[j], 0)
                j += 1
            yield f, name.group(1), src[i + 1:j - 1]


CHAINED = [(f, n, b) for f, n, b in kernels() if "pdl_begin(" in b]


def test_the_chain_was_found():
    assert {"k_gram_tc", "k_lincomb_tc", "k_cg_update", "k_tc_coef"} <= {n for _, n, _ in CHAINED}


@pytest.mark.parametrize("f,name,body", CHAINED, ids=[n for _, n, _ in CHAINED])
def test_tensor_memory_before_dependents(f, name, body):
    assert "pdl_wait(" in body
    if "tmem_alloc(" not in body:
        return
    a, b = body.index("tmem_alloc("), body.index("pdl_begin(")
    assert a < b, f"{f}: {name} lets dependents start before it has its tensor memory"
    between = body[a:b]
    assert "__syncthreads()" in between or "}" not in between, f"{f}: {name}: another warp may call pdl_begin before the allocation"
