"""What kernels that start under the tail of the one before them must keep to (csrc/common.h, launches), checked on their text:
the compiler cannot check it and no run shows it reliably."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_06629_b200", "csrc")


def _kernels():
    """{name: (parameters, body)} of every __global__ function."""
    found = {}
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, f)).read(), flags=re.S)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", text):
            def closing(at, opened, closed):
                depth = 1
                while depth:
                    depth += {opened: 1, closed: -1}.get(text[at], 0)
                    at += 1
                return at
            end = closing(m.end(), "(", ")")
            begin = text.index("{", end) + 1
            found[m.group(1)] = (text[m.end():end - 1], text[begin:closing(begin, "{", "}") - 1])
    return found


KERNELS = _kernels()
WAITING = sorted(name for name, (_, body) in KERNELS.items() if "launch_wait()" in body)


def test_every_kernel_launched_under_the_tail_of_another_waits():
    chained = set()
    for f in os.listdir(CSRC):
        if f.endswith((".cu", ".cuh")):
            for call in re.findall(r"(?:launch_chained\(|\bkernel = ).*?;", open(os.path.join(CSRC, f)).read(), flags=re.S):
                chained.update(k for k in KERNELS if re.search(r"\b%s\b" % k, call))
    assert len(chained) >= 10 and chained <= set(WAITING), chained - set(WAITING)


@pytest.mark.parametrize("name", WAITING)
def test_every_block_waits_before_it_leaves_or_lets_the_next_kernel_start(name):
    """A kernel is complete when its blocks are: one that leaves without waiting vouches for a kernel that may still run."""
    body = KERNELS[name][1]
    before = body[:body.index("launch_wait()")]
    before = re.sub(r"\[[&=]?\]\s*(\([^)]*\))?\s*\{[^{}]*\}", "", before)       # (a lambda's return is not the kernel's)
    assert "return" not in before and "launch_next()" not in before


@pytest.mark.parametrize("name", WAITING)
def test_nothing_lets_a_load_move_in_front_of_the_wait(name):
    """What the kernel before writes is no constant of the kernel that reads it: no restricted parameters, ..."""
    assert "__restrict__" not in KERNELS[name][0]


def test_no_read_only_loads():
    """... and no loads from the read-only path, in the kernels or in what they share."""
    for f in os.listdir(CSRC):
        if f.endswith((".cu", ".cuh", ".h")):
            assert not re.search(r"__ldg\s*\(|ld\.global\.nc", open(os.path.join(CSRC, f)).read()), f
