"""Kernels that start before the kernel in front of them has ended read what it
may have written by ordinary loads: the read-only path requires data that does
not change during the reading kernel's whole life, its time before the wait
included.  Checked on the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_11273_gb300", "csrc")


def _source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def _waiting_kernels():
    """(file, signature, body) of every kernel that waits for the kernel before it."""
    for name in sorted(os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cu"))):
        s = _source(name)
        for m in re.finditer(r"__global__[^;{}]*\)\s*\{", s):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(s[at], 0)
                at += 1
            if "wait_for_prerequisite()" in s[m.end():at]:
                yield name, m.group(0), s[m.end():at]


KERNELS = list(_waiting_kernels())


def test_every_waiting_kernel_is_found():
    calls = sum(_source(os.path.basename(p)).count("wait_for_prerequisite();")
                for p in glob.glob(os.path.join(CSRC, "*.cu")))
    assert len(KERNELS) == calls >= 5  # sort pass, reorder, table update, two traces


@pytest.mark.parametrize("k", range(len(KERNELS)))
def test_no_read_only_loads_in_waiting_kernels(k):
    name, signature, body = KERNELS[k]
    assert "__restrict__" not in signature, (name, signature)
    assert "__ldg(" not in body and ".nc" not in body, (name, signature)


def test_reorder_has_no_read_only_loads():
    s = _source("rr_permute.cu")  # its helpers included
    assert not re.search(r"__ldg\(|__restrict__|\.nc\b", s)


def test_trace_read_only_loads_are_of_the_bvh():
    s = _source("rr_trace.cu")
    assert "__restrict__" not in s
    for m in re.finditer(r"__ldg\(", s):
        assert re.match(r"__ldg\(&?(tp->|a\.tris\[)", s[m.start():]), s[m.start():m.start() + 60]
    # one read-only load in assembly, used for nodes and triangles only
    assert re.findall(r"ld\.global\.nc\.([\w:.]+)", s) == ["v8.b32"]
    for m in re.finditer(r"load256\(", s):
        assert re.match(r"load256\((np|&np->\w+|tp|const void \*p)\)", s[m.start():]), s[m.start():m.start() + 60]
