"""Chained launches (csrc/launch.cuh): a kernel's CTAs may be resident while the
kernel before it still writes, so what that kernel writes must not be read through
the read-only path (__ldg), whose data must not change while the reader lives.
Checked on the source: none of these loads depends on a GPU."""

from __future__ import annotations

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1905_00565_gb300", "csrc")


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def ldg_arguments(text):
    """The argument of every __ldg call, parentheses balanced."""
    for m in re.finditer(r"__ldg\(", text):
        depth, at = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[at], 0)
            at += 1
        yield text[m.end():at - 1]


# per file: the arrays that the kernel before may write, and the pointers derived
# from them (rho_kernel: the search's sums; table build: the points, boxes and
# sample of table_points_kernel; scans: the words of member_words_kernel)
WRITTEN_BEFORE = {
    "knn_dispatch.cu": ["partials", "base"],
    "table_build.cu": ["points", "pts", "box", "sbox", "smp", "src", "b", "c"],
    "knn_scan.cu": ["words", "src"],
    "row_walk.cuh": ["words"],
    "order.cu": ["series", "s"],
    "sampler.cu": ["order", "ord", "bits", "src"],
    "noalloc.cu": ["scratch"],
}


@pytest.mark.parametrize("name", sorted(WRITTEN_BEFORE))
def test_no_read_only_loads_of_what_the_kernel_before_writes(name):
    for arg in ldg_arguments(code(name)):
        used = set(re.findall(r"(?<![.>\w])[A-Za-z_]\w*", arg))
        assert not used & set(WRITTEN_BEFORE[name]), f"{name}: __ldg({arg})"


def test_every_chained_kernel_waits_before_it_reads():
    """chain_begin() stands before the first use of a kernel's pointers."""
    launched = set()
    for name in os.listdir(CSRC):
        for m in re.finditer(r"__global__.*?(\w+_kernel)\((.*?)\)\s*\{(.*?)\n\}", code(name), re.S):
            kernel, params, body = m.groups()
            if "plain" in kernel or "convergence" in kernel:   # plain launches
                continue
            assert "chain_begin();" in body, kernel
            before = body.split("chain_begin();")[0]
            pointers = re.findall(r"\*\s*(\w+)", params) + (["p"] if "Params" in params else [])
            for ptr in pointers:
                assert not re.search(rf"(?<![.>\w]){ptr}\s*(\[|->|\.)", before), (kernel, ptr)
            launched.add(kernel)
    assert len(launched) >= 9
