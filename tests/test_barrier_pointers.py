"""Shared-memory pointers around barriers in the transform passes.

`__restrict__` tells the compiler that during the function nothing else modifies the memory, so that a load
may move across a barrier after which it would see another thread's write.  A pass that contains such a
barrier (CTA, warp or named) therefore takes its field, tables and scratch without the qualifier.  Read
from the sources: a moved load shows in the generated code only.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_12686_gb300", "csrc")
BARRIER = re.compile(r"__syncthreads|__syncwarp|bar\.sync|row_sync\s*\(\)")


def _block(text, start, opening, closing):
    """End of the bracketed piece that opens at text[start]."""
    depth = 0
    for i in range(start, len(text)):
        depth += (text[i] == opening) - (text[i] == closing)
        if depth == 0:
            return i + 1
    raise ValueError("unbalanced source")


def _functions(text):
    """(name, parameters, body) of each __device__ function, member functions among them."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__device__[\w\s:<>,&*]*?\b(\w+)\s*\(", text):
        p1 = _block(text, m.end() - 1, "(", ")")
        body = re.match(r"[\s\w]*\{", text[p1:])
        if body:
            b0 = p1 + body.end() - 1
            yield m.group(1), text[m.end():p1 - 1], text[b0:_block(text, b0, "{", "}")]


@pytest.mark.parametrize("name", ["fft_block.cuh", "fft_block4.cuh"])
def test_no_restrict_across_a_barrier(name):
    with open(os.path.join(CSRC, name)) as f:
        found = list(_functions(f.read()))
    with_barrier = [(n, params) for n, params, body in found if BARRIER.search(body)]
    assert len(with_barrier) >= (1 if name == "fft_block.cuh" else 3)
    assert not [n for n, params in with_barrier if re.search(r"float2\s*\*\s*__restrict__", params)]
