"""The contract of the kernels' bounded waits, read off their sources (no GPU): the compute warps
meet named barriers inside their item loop, so a wait that ran out in some of them must be reduced
over all before a thread goes into the loop, or round it, on its own `failed` flag.  One that skips
the loop alone leaves the others at a barrier without a limit, which cannot be tried on a GPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_33591_gb300", "csrc")
FILES = ["kint_fwd.cu", "kint_fwd_main.cuh", "kint_bwd.cu", "kint_bwd_kv.cuh", "kint_bwd_fused.cu", "kint_probe.cu"]


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def closing(text, at):
    """The end of the bracketed region that opens at text[at]."""
    pairs, depth = {"(": ")", "{": "}"}, 0
    for k in range(at, len(text)):
        depth += (text[k] == text[at]) - (text[k] == pairs[text[at]])
        if depth == 0:
            return k
    raise AssertionError("unbalanced")


ASSIGN = re.compile(r"\bfailed\s*(?:\|=|=)(?!=)\s*([^;]+);")


def last_value(text):
    found = ASSIGN.findall(text)
    return found[-1] if found else None


@pytest.mark.parametrize("name", FILES)
def test_an_expired_wait_is_reduced_before_every_item_loop_and_round(name):
    text = code(name)
    loops = 0
    for m in re.finditer(r"\b(?:for|while)\s*\(", text):
        end = closing(text, m.end() - 1)
        if "p.nitems" not in text[m.start():end] or "!failed" not in text[m.start():end]:
            continue
        loops += 1
        body_at = text.index("{", end)
        start = text.rindex("bool failed", 0, m.start())
        before = last_value(text[start:m.start()])
        assert before == "false" or before.startswith("group_any"), (name, before)
        body = last_value(text[body_at:closing(text, body_at)])
        assert body.startswith("group_any"), (name, body)
    assert loops >= 1, name
