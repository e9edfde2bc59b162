"""Kernels launched with programmatic dependent launch are resident while the
kernel before them may still write what they read: they read global memory by
plain loads that stay behind the wait, never through the read-only path."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_10558_gb300", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def _body(src, at):
    """The brace block that follows position `at`."""
    i = src.index("{", at)
    depth = 0
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth == 0:
            return src[i:j + 1]
    raise AssertionError("unbalanced braces")


@pytest.mark.parametrize("name", FILES)
def test_no_read_only_loads(name):
    src = _code(name)
    assert not re.search(r"ld\.global\.nc|__ldg\s*\(", src), name
    # inline loads are ordered against the wait and the barriers
    for m in re.finditer(r"asm\s*(volatile)?\s*\(\s*\"ld\.global", src):
        assert m.group(1) and '"memory"' in src[m.start():src.index(";\n", m.start())], name


def test_waiting_kernels_take_no_read_only_pointer():
    seen = 0
    for name in FILES:
        src = _code(name)
        for m in re.finditer(r"__global__[^;{]*?\b(\w+_kernel)\s*\(", src):
            body = _body(src, m.end())
            if "grid_wait()" not in body:
                continue
            seen += 1
            params = src[m.end():src.index("{", m.end())]
            assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", params + body), m.group(1)
        if name.endswith(".cuh"):  # what they share
            assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", src), name
    assert seen >= 12
