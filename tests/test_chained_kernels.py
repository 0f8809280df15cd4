"""What chained launches ask of a kernel (csrc/gm_launch.cuh), read from the sources: it waits for its
predecessor before anything else, and none of its loads takes memory for read-only."""
import os
import re

import paper_2410_17133_gb300 as gm

CSRC = os.path.join(os.path.dirname(gm.__file__), "csrc")


def code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


SOURCES = {n: code(n) for n in sorted(os.listdir(CSRC)) if n.endswith((".cu", ".cuh"))}


def test_no_load_takes_memory_for_read_only():
    for name, text in SOURCES.items():
        assert not re.search(r"__ldg\b|__restrict__|\bld\.global(\.\w+)*\.nc\b|__ldlu\b", text), name


def test_chained_kernels_wait_first():
    kernels = 0
    for name, text in SOURCES.items():
        for m in re.finditer(r"(\w+)\(int chained[^{;]*\)\s*\{\s*([^;]*;)", text):
            if m.group(1) == "gm_chain":
                continue
            kernels += 1
            assert m.group(2).strip() == "gm_chain(chained);", (name, m.group(1))
    assert kernels >= 20
