"""Inline assembly that exchanges values between lanes is volatile.

An asm statement without `volatile` is a pure function of its operands to the
compiler, which may then merge, move or sink it, for a .sync instruction into
code that not all lanes of its mask run.
"""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sync_instructions_are_volatile():
    seen = 0
    for path in glob.glob(os.path.join(ROOT, "paper_1704_04381_gb300", "csrc", "*.cu*")):
        with open(path) as f:
            text = f.read()
        for m in re.finditer(r"\basm\b\s*(volatile|__volatile__)?\s*\(([^;]*?;[^;]*?)\)\s*;", text):
            if ".sync" in m.group(2):
                seen += 1
                assert m.group(1), (os.path.basename(path), m.group(0))
    assert seen
