"""A kernel that may start beside the one before it reads that kernel's results by plain loads.

Read-only loads (__ldg) are for data that nothing writes while the kernel lives, and the compiler may
move them ahead of the wait for the kernel before; the call's own scratch is no such data."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0907_3768_gb300", "csrc")
# the arrays that a call's kernels write for one another: absorbed powers, ordering, pairs, records, partial sums
SCRATCH = r"\b(S|Srow|key|bkt|hist|order|prep|cell|part|accp|Jw|Lprev)\b\s*(\+|\)|\[|->|\.)"


def test_scratch_is_not_read_through_the_read_only_path():
    bad = []
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"__ldg\(", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[end], 0)
                end += 1
            arg = text[m.end():end]
            pointer = re.split(r"\+", re.sub(r"reinterpret_cast<[^>]*>", "", arg))[0] + "+"
            if re.search(SCRATCH, pointer):
                bad.append(f"{name}: __ldg({arg}")
    assert not bad, bad
