"""A verification whose bounded wait runs out must not leave path_len and bonus_token as the allocator gave them: a stale
length and token look like a result.  No input makes a wait run out, so this reads the kernels: every exit behind a wait
goes through the function that writes 0 and -1, and that function does."""
import os
import re

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_12374_b200", "csrc", "tree_verify_walk.cu")


def test_every_exit_behind_a_wait_leaves_defined_results():
    text = open(SOURCE).read()
    kernels = text[text.index("tree_verify_walk_kernel(const VerifyArgs a_in)"):]
    waits = [line for line in kernels.splitlines() if re.search(r"!(exchange_pull<|bar_wait)", line)]
    assert len(waits) >= 5  # two in the default walk, one in the greedy one, two in the sampling one
    for line in waits:
        assert re.search(r"\) return timed_out\(a\);", line), line
    body = text[text.index("void timed_out("):]
    body = body[:body.index("\n}")]
    assert "*a.path_len = 0;" in body and "*a.bonus = -1;" in body
