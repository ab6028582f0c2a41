"""All work of a call is on the caller's stream (include/evap.h): no copy, clearing or launch of the library goes to the
legacy default stream, which does not order work before that of a non-blocking stream (no GPU needed: the sources)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2401_07805_gb300", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("name", FILES)
def test_copies_and_clears_name_a_stream(name):
    assert re.findall(r"\bcuda(?:Memset|Memcpy|MemcpyToSymbol|MemcpyFromSymbol)\s*\(", code(name)) == []


@pytest.mark.parametrize("name", FILES)
def test_launches_name_a_stream(name):
    src = code(name)
    starts = [m.end() for m in re.finditer("<<<", src)]
    for a in starts:
        args, depth = [""], 0
        for ch in src[a:src.index(">>>", a)]:
            depth += (ch in "([{") - (ch in ")]}")
            if ch == "," and depth == 0:
                args.append("")
            else:
                args[-1] += ch
        assert len(args) == 4 and args[3].strip() in ("s", "st", "c.s"), src[a - 60:a + 80]
