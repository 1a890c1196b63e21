"""Which lanes wait and commit in the tensor-core kernels, read from the sources (no GPU needed).

A commit covers only the products of the thread that executes it, so a warp that issues them from an elected lane must
commit from the elected lane too, also where it waits for what is in flight after a timeout.  And no lane may leave a loop that
its warp meets in (an election, a warp barrier) because its own wait gave up: the others would wait for it without end.
It stays and waits no more (`ok = ok && mbar_wait(..)`), or the warp votes (`warp_wait`)."""
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


@pytest.mark.parametrize("name", ["attn.cu", "image_tc.cu"])
def test_no_lane_leaves_its_warp_after_a_wait(name):
    text = open(os.path.join(CSRC, name)).read()
    lines = [line.split("//")[0] for line in text.splitlines()]
    elected = {no for no, conditions in guarded_calls(text, "mbar_wait") if any("elect_one()" in c for c in conditions)}
    for no, code in enumerate(lines, 1):
        if "mbar_wait(" not in code or "__device__" in code or "(void)mbar_wait(" in code or no in elected:
            continue
        kept = re.search(r"\b(ok|mma_ok) = ((ok|s_fail == 0) && )?mbar_wait\(|__all_sync\(0xFFFFFFFFu, mbar_wait\(", code)
        assert kept, f"{name}:{no}: {code.strip()}"
        assert not re.search(r"if \(!ok\)|break", " ".join(lines[no:no + 2])), f"{name}:{no}: leaves after its own wait"
