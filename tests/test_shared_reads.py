"""Reads of shared memory by inline assembly are ordered where they have to be.

A plain `asm` load is a function of its address to the compiler: nothing keeps
it behind a barrier or before a store to the same place. So the functions that
read a unit's header, descriptors and column ends, row sums or slots (memory
that is written again and again at one address) use the ordered helpers, and an
ordered helper is `asm volatile` with a memory clobber. CPU only (source text)."""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_02893_gb300", "csrc")
PLAIN = re.compile(r"\blds_(?!volatile)\w*?(?<!_ordered)(?:<[^>]*>)?\s*\(")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def body(text, function):
    """The body of the one function (or kernel) of that name."""
    found = [m for m in re.finditer(rf"\b{function}\s*\(", text)]
    for m in found:
        i, depth = m.end(), 1
        while depth:                                   # the parameter list
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        if not text[i:].lstrip().startswith("{"):
            continue                                   # a call or a declaration
        i = start = text.index("{", i) + 1
        depth = 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        return text[start:i]
    raise AssertionError(f"{function} not found")


@pytest.mark.parametrize("name,function", [
    ("vbq_gemm.cu", "consume_unit_b"), ("vbq_gemm.cu", "flush_rows"), ("vbq_gemm.cu", "flush_cluster"),
    ("vbq_gemm.cu", "gemmb_kernel"), ("vbq_gemv.cu", "consume_unit"), ("vbq_gemv.cu", "consume_single_w"),
    ("vbq_gemv.cu", "build_tables"), ("vbq_gemv.cu", "team_flush"), ("vbq_gemv.cu", "gemv1_kernel"),
    ("vbq_gemv.cu", "gemv1_unit_kernel"), ("vbq_gemv.cu", "gemv_chain_kernel")])
def test_reads_behind_barriers_are_ordered(name, function):
    assert PLAIN.findall(body(source(name), function)) == []


def test_ordered_helpers_cannot_be_moved():
    text = source("vbq_device.cuh")
    names = re.findall(r"\b(lds_\w*(?:_ordered|_volatile)|lds_volatile)\s*\(", text)
    assert "lds_f32x4_ordered" in names and "lds_volatile" in names
    for n in set(names):
        b = body(text, n)
        assert "asm volatile" in b and '"memory"' in b, n
    for name in os.listdir(CSRC):                      # defined nowhere else
        if name.endswith((".cu", ".cuh", ".h")) and name != "vbq_device.cuh":
            assert not re.search(r"__forceinline__[^\n;{]*\blds_\w*_ordered\s*\(", source(name)), name
