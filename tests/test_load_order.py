"""Loads written in PTX stay behind a kernel's wait for its predecessor.

A kernel launched as a programmatic dependent runs beside the kernel before it
until its griddepcontrol.wait.  The compiler keeps volatile asm statements in
order and may move others, so every asm that loads global memory has to be
volatile (or clobber memory), like the wait itself."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1502_02389_gb300", "csrc")


def test_global_loads_in_asm_are_volatile():
    loads = 0
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        with open(os.path.join(CSRC, f)) as fh:
            text = fh.read()
        for m in re.finditer(r"\basm\s*(volatile)?\s*\((.*?)\)\s*;", text, re.S):
            if re.search(r"\bld\.global|\bld\.relaxed|\bcp\.async|griddepcontrol", m.group(2)):
                loads += "ld.global" in m.group(2)
                assert m.group(1), (f, m.group(2)[:80])
    assert loads >= 5
