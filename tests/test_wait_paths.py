"""What the tensor-core kernels do after a bounded wait has run out, read from
their sources (no GPU test makes a wait inside them run out)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1002_0916_gb300", "csrc")
SOURCES = ("sep32.cu", "umma.cu", "umma2.cu", "umma_gen.cu")


def _statements(text):
    """(statement or block header, headers of the blocks around it) in order."""
    text = re.sub(r"//[^\n]*", "", text)
    out, around, cur, paren = [], [], "", 0
    for ch in text:
        paren += {"(": 1, ")": -1}.get(ch, 0)
        if ch in "{};" and not (ch == ";" and paren):
            out.append((" ".join(cur.split()), tuple(around)))
            if ch == "{":
                around.append(out[-1][0])
            elif ch == "}":
                around.pop()
            cur = ""
        else:
            cur += ch
    return out


@pytest.mark.parametrize("name", SOURCES)
def test_the_abort_flag_is_voted_on(name):
    """Another warp can set the flag at any time, and the loads of tensor memory,
    shuffles and barriers want whole warps: every read of it is one lane's alone
    or goes through a vote."""
    with open(os.path.join(CSRC, name)) as fh:
        stmts = _statements(fh.read())
    reads = [(s, around) for s, around in stmts
             if "abort_flag" in s and not re.search(r"abort_flag( = [01])?$", s)]
    assert reads
    for s, around in reads:
        assert "__all_sync(" in s or any("lane == 0" in h for h in (s, *around)), s
