"""The one-warp instance of the per-group resampler, by its source: a lane
zeroes marks that other lanes then set, and reads marks that other lanes set,
so a barrier has to lie between those accesses in the code that TEAM == 32
compiles (shuffles order no memory between lanes).  A race shows itself on no
result as long as the lanes happen to run together, so the order is checked
here and the results in test_gpu_resample_groups.py."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1310_4624_gb300", "csrc",
                   "pf_kernels.cu")


def _block(text, at):
    """End of the brace block that opens at or after `at`."""
    i = text.index("{", at)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return j + 1
    raise AssertionError("unbalanced braces")


def _one_warp_body():
    """k_resample_groups as TEAM == 32 compiles it: comments, the lambdas and
    the branches of larger teams taken out."""
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    start = text.index("k_resample_groups(const")
    body = text[start:_block(text, start)]
    for opener in (r"auto (?:sync|scan|item0) = \[", r"if constexpr \(TEAM > 32\) \{"):
        while True:
            m = re.search(opener, body)
            if not m:
                break
            end = _block(body, m.start())
            body = body[:m.start()] + body[end:]
    return body


ZERO = r"make_uint4\(0u, 0u, 0u, 0u\)"
MARK = r"s_mark\[pos\] ="
READ = r"m\[r\] = q\.x"
BARRIER = r"(?<![_\w])sync\(\);|__syncwarp\(\);"


def test_initial_clear_and_first_marks_are_ordered():
    body = _one_warp_body()
    zero, mark = re.search(ZERO, body), re.search(MARK, body)
    assert zero and mark and zero.start() < mark.start()
    assert re.search(BARRIER, body[zero.end():mark.start()]), "no barrier between clearing the marks and setting them"


@pytest.mark.parametrize("first,then", [(MARK, READ), (READ, r"store_items<ITEMS>")])
def test_windows_are_ordered(first, then):
    """Marks set, then read and cleared, then (next window) set again."""
    body = _one_warp_body()
    a = re.search(first, body)
    b = re.search(then, body[a.end():])
    assert re.search(BARRIER, body[a.end():a.end() + b.start()])
