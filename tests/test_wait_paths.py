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


@pytest.mark.parametrize("name,kernels", [("sep32.cu", 1), ("umma2.cu", 2), ("umma.cu", 2),
                                          ("umma_gen.cu", 1)])
def test_a_timeout_waits_for_the_mmas_in_flight(name, kernels):
    """Every kernel that issues MMAs commits them once more after its loop over
    the K blocks, to a barrier that its CTA waits on before tensor memory is
    released: the accumulator's in the one-tile kernels, `drain` (where a wait
    ran out) in the persistent ones, whose epilogue may have left."""
    with open(os.path.join(CSRC, name)) as fh:
        bodies = fh.read().split("__global__")[1:]
    bodies = [b for b in bodies if re.search(r"\bmma2?_f16\(", b)]
    assert len(bodies) == kernels
    for b in bodies:
        bar = "drain" if "uint64_t acc_full" in b else "accum_bar"
        last_mma = max(m.end() for m in re.finditer(r"\bmma2?_f16\(", b))
        commit = [m.end() for m in re.finditer(r"commit2?\(&" + bar, b) if m.end() > last_mma]
        waits = [m.end() for m in re.finditer(r"wait\w*\(&" + bar + ", 0", b)]
        release = b.index("tmem_dealloc")
        assert commit and any(commit[-1] < w < release for w in waits), bar
        if bar == "drain":
            assert re.search(r"if \(!ok\) \{[^}]*commit2?\(&drain[^}]*wait\w*\(&drain", b)
