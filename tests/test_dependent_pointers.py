"""Kernels that start before the previous one on the stream has ended (those that
call pdl_wait) must not take what that one writes through const __restrict__
pointers: such loads may be moved ahead of the wait or go through the
non-coherent path.  Read from the sources (no GPU)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2201_03950_gb300", "csrc")
# complete before the kernel's predecessor starts, see the kernel
COMPLETE = {"k_varlen_solve": {"a", "b", "c"}}


def kernels(text):
    """(name, parameters, body) of every __global__ function of a source."""
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
        i = j = m.end()
        depth = 1
        while depth:
            depth += {"(": 1, ")": -1}.get(text[j], 0)
            j += 1
        k = e = text.index("{", j) + 1
        depth = 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[e], 0)
            e += 1
        yield m.group(1), text[i:j - 1], text[k:e]


def waiting():
    for f in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for name, params, body in kernels(text):
            if "pdl_wait()" in body:
                yield pytest.param(name, params, id=name)


def test_the_waiting_kernels_are_found():
    names = {p.id for p in waiting()}
    assert {"k_varlen_solve", "k_strided_tma", "k_strided", "k_chunk_cluster", "k_lines_tma",
            "k_adi_planes", "k_adi_zlines", "k_adi_zw", "k_v2_rhs_adj4"} <= names


@pytest.mark.parametrize("name,params", list(waiting()))
def test_no_restricted_reads(name, params):
    found = set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params))
    assert found <= COMPLETE.get(name, set())
