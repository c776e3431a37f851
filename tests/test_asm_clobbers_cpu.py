"""Inline assembly that reads or writes memory the compiler also accesses
(asynchronous copies into shared memory, the waits that order them) must say
so with a "memory" clobber; without it the compiler may move other accesses
of the same shared memory across the statement."""
import glob
import os
import re

import paper_2605_14780_gb300 as pkg

CSRC = os.path.join(os.path.dirname(os.path.abspath(pkg.__file__)), "csrc")
TOUCHES = ("cp.async", "griddepcontrol.wait", "st.", "ld.", "red.", "atom.")


def _statements():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        with open(path) as f:
            text = f.read()
        for m in re.finditer(r"\basm(?:\s+volatile)?\s*\((.*?)\)\s*;", text, re.S):
            yield os.path.basename(path), m.group(0)


def test_memory_instructions_carry_the_clobber():
    found = [s for s in _statements() if any(t in s[1] for t in TOUCHES)]
    assert found
    for name, stmt in found:
        assert '"memory"' in stmt and "volatile" in stmt, f"{name}: {stmt}"
