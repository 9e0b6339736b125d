"""How the kernels wait on a barrier, read from their source (no GPU): every lane polls with its own clock, so after a wait by a
whole warp its lanes may disagree about whether it was met.  Either the warp votes, or the wait is mbar_wait_stay, after which a
lane that gave up goes on with the others."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_20332_b200", "csrc")
ONE_THREAD = re.compile(r"\blane == 0|threadIdx\.x == 0")


def waits(text):
    """(line, innermost-first opening lines of the blocks around it, the three lines from it on) of each bare mbar_wait call."""
    lines = [re.sub(r"//.*", "", line) for line in text.splitlines()]
    stack, out = [], []
    for i, line in enumerate(lines):
        if re.search(r"\bmbar_wait(_cluster)?\(", line) and "__device__" not in line:
            out.append((i + 1, list(stack), " ".join(lines[i:i + 3])))
        for ch in line:
            if ch == "{":
                stack.append(line)
            elif ch == "}":
                stack.pop()
    return out


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_a_waiting_warp_agrees(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    for line, blocks, after in waits(text):
        one_thread = any(ONE_THREAD.search(b) for b in blocks)
        assert one_thread or "__all_sync" in after, f"{name}:{line}: a whole warp waits and goes on with lanes that may disagree"


def test_the_check_itself():
    bad = "if (warp > 3) {\n  if (!(ok = mbar_wait(b, 0, f))) break;\n  tc_fence_after();\n  tmem_ld32(t, v);\n}"
    good = "if (lane == 0) {\n  if (!(ok = mbar_wait(b, 0, f))) break;\n}"
    for text, fine in ((bad, False), (good, True)):
        (_, blocks, after), = waits(text)
        assert (any(ONE_THREAD.search(b) for b in blocks) or "__all_sync" in after) == fine
