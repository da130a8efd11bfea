"""Kernels launched by programmatic dependent launch start before the previous kernel's words are visible: what
they read of them has to be a plain load through a plain pointer (ld.global.nc is for data that is constant for
the kernel's whole life, and __restrict__ lets a load move above the wait).  Checked in the sources: __ldg is
left for the context's tables, and no operand pointer is __restrict__."""
import os
import re

import pytest

from paper_1908_06972_gb300 import _build

# the context's tables (primes, twiddles, conversion constants) and the key words of k_ks_inner_bulk, written
# launches before (at least the transforms of the digits lie between)
TABLES = re.compile(r"&t\.|&tw\[|&tab\[|&T\[|&J\.table\[|&J\.tc\[|&cs\[|&consts\[|&lm\[|p[ab]\)|reinterpret_cast<const ulonglong2\*>\(p[ab]\)")


def functions(name):
    """(head, body) of every function of a source file."""
    with open(os.path.join(_build.CSRC, name)) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    for m in re.finditer(r"^(?:template[^\n]*\n)?(?:__global__|__device__)[^;{]*\{", src, re.M):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        yield m.group(0), src[m.end():i]


def dependent(name):
    return [(h, b) for h, b in functions(name) if "pdl_wait()" in b or "fwd_rows<" in b]


@pytest.mark.parametrize("name,least", [("ntt.cu", 4), ("poly.cu", 7)])
def test_operands_are_plain_loads(name, least):
    found = dependent(name)
    assert len(found) >= least
    for head, body in found:
        for arg in re.findall(r"__ldg\(([^;]*)", body):
            assert TABLES.match(arg), (head, arg)
        assert "__restrict__" not in head and "__restrict__" not in body, head
