"""PTX leaves the destination registers of tcgen05.ld undefined until tcgen05.wait::ld.  A read before the wait shows in no result
as long as the compiler happens to schedule it late, so the kernels' source is read instead: between a load into an array and the
next wait, nothing in the same block names the array."""
from __future__ import annotations

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_25188_b200", "csrc")
LOAD = re.compile(r"tmem_ld_x(?:16|32)\(([^;]*)\);|tmem_load_cols\(([^;]*)\);")


def reads_before_the_wait(text):
    """[(array, line)] of every mention of a load's array ahead of the wait.  A load under an `if` without braces belongs to the block
    around it; the scan ends with that block, where the order of the text is no longer the order of execution."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", lambda m: re.sub(r"[^\n]", " ", m.group(0)), text, flags=re.S)
    found = []
    for m in LOAD.finditer(text):
        args = m.group(1) or m.group(2)
        array = re.match(r"\s*(\w+)", args.split(",")[1]).group(1)
        depth, end = 0, m.end()
        while end < len(text) and depth >= 0 and not text.startswith("tmem_ld_wait()", end):
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
        between = LOAD.sub(lambda q: " " * len(q.group(0)), text[m.end():end])   # a further load into it is no read, nor is a member of that name
        for use in re.finditer(r"(?<![.\w])%s\b" % array, between):
            found.append((array, text.count("\n", 0, m.end() + use.start()) + 1))
    return found


def test_the_check_sees_a_copy_ahead_of_the_wait():
    bad = "for (;;) { tmem_ld_wait(); if (more) ptx::tmem_ld_x16(t + c, vn); use(v); for (i) v[i] = vn[i]; }"
    good = "ptx::tmem_ld_x16(t, va); for (;;) { tmem_ld_wait(); ptx::tmem_ld_x16(t + c, vb); use(va); tmem_ld_wait(); use(vb); }"
    assert [a for a, _ in reads_before_the_wait(bad)] == ["vn"]
    assert reads_before_the_wait(good) == []


@pytest.mark.parametrize("name", sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu*"))))
def test_no_register_of_a_tensor_memory_load_is_read_before_its_wait(name):
    assert reads_before_the_wait(open(os.path.join(CSRC, name)).read()) == []
