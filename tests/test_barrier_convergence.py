"""Warp convergence before the .aligned instructions whose callers may arrive
diverged, by reading the sources: a warp whose lanes execute one of them apart is
undefined behaviour, which no run shows reliably and none should provoke."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2609_36835_gb300" / "csrc"


@pytest.mark.parametrize("instruction", [r"barrier\.cluster\.(?:arrive|wait)", r"tcgen05\.alloc", r"tcgen05\.dealloc"])
def test_aligned_instructions_follow_a_syncwarp(instruction):
    found = 0
    for src in sorted(CSRC.glob("*.cu*")):
        for m in re.finditer(r'asm volatile\(\s*"' + instruction, src.read_text()):
            found += 1
            before = src.read_text()[:m.start()].rstrip()
            line = before.count("\n") + 2
            assert before.endswith("__syncwarp();"), "%s:%d" % (src.name, line)
    assert found
