"""Loads of the kernels' sources.

A kernel launched as a programmatic dependent is resident while its
predecessor still writes the links, so no load of device memory may take the
read-only path (__ldg, ld.global.nc): that one is right only for memory that
nothing writes for the kernel's whole lifetime, and may be moved before the
wait for the predecessor.  Nothing on a GPU shows the difference reliably, so
the rule is checked where it is written."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_0904_0642_gb300", "csrc")


def test_no_load_takes_the_read_only_path():
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh", ".h")):
            continue
        with open(os.path.join(CSRC, name)) as f:
            code = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
        seen += len(re.findall(r"\bld_link<", code))
        assert not re.search(r"__ldg\b|\.nc\b", code), name
        # the compiler chooses that path by itself for const __restrict__ pointers
        assert "__restrict__" not in code, name
    assert seen > 10
