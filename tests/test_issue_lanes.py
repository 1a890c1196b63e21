"""Which lane commits tensor-core work, read from the sources (no GPU needed): a commit covers only the products of
the thread that executes it, so a warp that issues them from an elected lane must commit from the elected lane too, also
where it waits for what is in flight after a timeout."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_02612_gb300", "csrc")


def guarded_calls(text, name):
    """(line number, innermost enclosing conditions) of every call of `name`, by braces."""
    stack, calls = [], []
    for no, line in enumerate(text.splitlines(), 1):
        code = line.split("//")[0]
        if re.search(rf"\b{name}\(", code) and "__device__" not in code:
            calls.append((no, [c for c in stack if "if" in c]))
        for ch in re.findall(r"[{}]", code):
            if ch == "{":
                stack.append(code.strip())
            elif stack:
                stack.pop()
    return calls


@pytest.mark.parametrize("name", ["attn.cu", "image_tc.cu"])
def test_commits_come_from_the_elected_lane(name):
    calls = guarded_calls(open(os.path.join(CSRC, name)).read(), "umma_commit")
    assert len(calls) >= 3, "the sources moved"
    for no, conditions in calls:
        assert any("elect_one()" in c for c in conditions), f"{name}:{no}: a commit from a lane that was not elected"
