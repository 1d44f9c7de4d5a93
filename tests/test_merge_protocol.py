"""The word through which the CTAs of a head settle who merges a share of its rows: every order in which
a few CTAs can arrive, give their shares up and be the last one.  Each share is merged once and the word
ends as it began, provided that a CTA's own arrival is in the word before it gives up; that order
is what the two fences around the arrival flag in the kernel are for."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_05650_b200", "csrc",
                   "verify_attn_tc.cu")


def outcomes(n, ordered, tries=2):
    """(merges of each share, word at the end) over all orders of the steps of n CTAs.  A CTA: its arrival
    (0 to come, 1 counted, 2 counted as the last: shares it saw given up are merged, the word goes back to zero
    a step later, 3 done); its own share (0 undecided, 1 given up and seen by nobody or too late: keeps it, but has
    its bit to take back, 2 handed over, 3 merged by itself); give-ups so far."""
    seen, ends = set(), set()
    stack = [((0,) * n, (0,) * n, (0,) * n, (0, 0), (0,) * n)]
    put = lambda t, i, x: t[:i] + (x,) + t[i + 1:]
    while stack:
        state = stack.pop()
        if state in seen:
            continue
        seen.add(state)
        arr, own, gave, (count, bits), merged = state
        nxt = []
        for i in range(n):
            if arr[i] == 0:
                if count + 1 < n:
                    nxt.append((put(arr, i, 1), own, gave, (count + 1, bits), merged))
                else:
                    m = tuple(k + (bits >> j & 1) for j, k in enumerate(merged))
                    nxt.append((put(arr, i, 2), own, gave, (n, bits), m))
            elif arr[i] == 2:
                nxt.append((put(arr, i, 3), own, gave, (0, 0), merged))
            if own[i] == 0 and all(arr):                       # every partial is there
                nxt.append((arr, put(own, i, 3), gave, (count, bits), put(merged, i, merged[i] + 1)))
            if own[i] == 0 and gave[i] < tries and (arr[i] or not ordered):
                word = (count, bits | 1 << i)
                nxt.append((arr, put(own, i, 1 if count == 0 else 0 if count >= n else 2), put(gave, i, gave[i] + 1),
                            word, merged))
            if own[i] == 1:                                    # a count of zero: all have arrived, take the bit back
                nxt.append((arr, put(own, i, 0), gave, (count, bits & ~(1 << i)), merged))
        if not nxt:
            ends.add((merged, (count, bits)))
        stack += nxt
    return ends


@pytest.mark.parametrize("n", [2, 3])
def test_each_share_is_merged_once(n):
    assert outcomes(n, True) == {((1,) * n, (0, 0))}


def test_a_give_up_ahead_of_the_own_arrival_can_merge_a_share_twice():
    assert any(max(merged) > 1 for merged, _ in outcomes(2, False))


def test_the_kernel_orders_the_arrival():
    code = re.sub(r"//[^\n]*", "", open(SRC).read())
    assert re.search(r"atomicAdd\(word, 1ull\);.*?__threadfence_block\(\);\s*\*arrived_s = 1;", code, flags=re.S)
    assert re.search(r"if \(\*arrived_s\) \{\s*__threadfence_block\(\);[^}]*?atomicOr\(word, bit\)", code, flags=re.S)
    assert len(re.findall(r"\*arrived_s = 1", code)) == 1
