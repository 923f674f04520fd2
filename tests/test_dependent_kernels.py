"""Kernels that are launched while the launch before them drains read what it
wrote only after their wait.  A load through a __restrict__ pointer may be moved
before launch_wait() (no other access is said to alias it), so such kernels take
no __restrict__ pointers, or take their block index from launch_wait_block(), on
which every address then depends."""
import os
import re

from paper_2007_12908_gb300 import build

KERNEL = re.compile(r"__global__[^;{]*?\b(k_\w+)\s*\(([^{;]*)\)\s*\{", re.S)


def _body(src, start):
    depth = 1
    for i in range(start, len(src)):
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        if depth == 0:
            return src[start:i]
    raise AssertionError("unbalanced braces")


def _kernels():
    for name in sorted(os.listdir(build.CSRC)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, name)).read())
        for m in KERNEL.finditer(src):
            yield name, m.group(1), m.group(2), _body(src, m.end())


def test_restrict_pointers_wait():
    waiting = blocks = 0
    bad = []
    for name, kernel, params, body in _kernels():
        if "launch_wait_block()" in body:
            blocks += 1
            # the only block index is the one that is known after the wait
            if "blockIdx" in body:
                bad.append(f"{name}: {kernel} reads blockIdx")
        elif "launch_wait()" in body:
            waiting += 1
            if "__restrict__" in params + body:
                bad.append(f"{name}: {kernel}")
    assert waiting >= 10 and blocks >= 5  # the pattern finds them
    assert not bad, bad
