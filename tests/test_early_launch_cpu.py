"""Loads of what an earlier launch writes, in the kernels that launch_early may
start before that launch has ended (read from the sources, no GPU): an inline
global load is volatile with a memory clobber, so that it stays after
wait_for_previous, and is not .nc, which is for data that nothing writes while
the kernel lives."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2111_05651_gb300", "csrc")
FILES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))


def _text(path):
    with open(path) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_inline_global_loads_are_ordered(path):
    for m in re.finditer(r"\basm\b(\s+volatile)?\s*\(((?:[^();]|\([^();]*\)|;(?=[^\n]*\"))*)\);", _text(path)):
        if "ld.global" not in m.group(2):
            continue
        assert m.group(1), f"not volatile: {m.group(0)}"
        assert '"memory"' in m.group(2), f"no memory clobber: {m.group(0)}"
        assert ".nc" not in m.group(2), f"read-only load: {m.group(0)}"


def test_every_inline_global_load_was_looked_at():
    asm = r"\basm\b(?:\s+volatile)?\s*\((?:[^();]|\([^();]*\)|;(?=[^\n]*\"))*\);"
    for path in FILES:
        text = _text(path)
        assert text.count("ld.global") == sum(s.count("ld.global") for s in re.findall(asm, text)), path

