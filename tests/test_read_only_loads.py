"""Which data the kernels read through the read-only path.

`__ldg` asks for data that no one writes while the kernel exists.  A kernel
launched to overlap its predecessor exists while that one still runs, so what
the predecessor writes must be read by ordinary loads after the wait.  The
arrays listed here are safe: the bond list never changes after the set-up, and
the flip bits are written two kernels before the one that reads them."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_08312_gb300", "csrc")
SAFE = ("G.bi", "G.bj", "bi", "bj", "R.F", "S.fb")


def read_only_arguments(text):
    """The argument of every __ldg( ... ) of a source text, comments left out."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    for m in re.finditer(r"\b__ldg\s*\(", text):
        depth, k = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[k], 0)
            k += 1
        yield text[m.end():k - 1]


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_read_only_loads_are_of_finished_arrays(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    for arg in read_only_arguments(text):
        base = re.sub(r"reinterpret_cast<[^>]*>\(", "", arg).split("+")[0].strip()
        assert base in SAFE, f"{name}: __ldg({arg})"
    assert "ld.global.nc" not in text and "__restrict__" not in text
