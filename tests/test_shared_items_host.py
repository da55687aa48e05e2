"""The blend backward's shared items: two warps of a pair take each claim from shared memory, written by the
even warp before a barrier of both.  Every order in which the two warps' steps can happen is run here, with
as many claim words per pair as the kernel has: both warps work on the same items, and both leave.  (An id
without a chunk sends both straight to the next claim, with no further barrier.)  On the host: the
order of two warps cannot be forced on a device, and a lost claim there would leave a warp waiting."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def claim_words():
    src = open(os.path.join(ROOT, "paper_2503_13086_gb300", "csrc", "k_blend.cu")).read()
    m = re.search(r"constexpr unsigned kClaimWords = (\d+);", src)
    if not m:
        return 1  # one word, rewritten by every claim
    assert "s_claim[kBwdWarps / 2][kClaimWords]" in src and "[turn % kClaimWords]" in src
    return int(m.group(1))


def outcomes(has_chunk, words):
    """All (items of the even warp, items of the odd warp) the protocol can end in; None: a warp waits for ever."""
    n = len(has_chunk)
    # a warp: (step, turn, ids worked on); steps: 0 store the claim (even only), 1 wait at the claim's
    # barrier, 2 read the claim, 3 wait at the item's barrier, 4 gone
    start = ((0, 0, ()), (1, 0, ()), (0,) * words, 0)  # even, odd, claim words, next id
    seen, todo, ends = {start}, [start], set()
    while todo:
        even, odd, claim, nxt = todo.pop()
        succ = []

        def put(w, st, claim=claim, nxt=nxt):
            succ.append(((st, odd) if w == 0 else (even, st)) + (claim, nxt))

        for w, (step, turn, got) in enumerate((even, odd)):
            if step == 0:
                c = list(claim)
                c[turn % words] = nxt
                put(w, (1, turn, got), tuple(c), nxt + 1)
            elif step == 2:
                i = claim[turn % words]
                first = 0 if w == 0 else 1
                if i >= n:
                    put(w, (4, turn, got))
                elif not has_chunk[i]:
                    put(w, (first, turn + 1, got))
                else:
                    put(w, (3, turn, got + (i,)))
        if even[0] in (1, 3) and odd[0] in (1, 3):  # a barrier does not know where in the code it was reached
            def past(w, st):
                return (2, st[1], st[2]) if st[0] == 1 else (0 if w == 0 else 1, st[1] + 1, st[2])
            succ.append((past(0, even), past(1, odd), claim, nxt))
        if not succ:
            ends.add((even[2], odd[2]) if even[0] == 4 and odd[0] == 4 else None)
        for s in succ:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return ends


@pytest.mark.parametrize("has_chunk", [(1, 1), (0, 1), (1, 0, 1), (0, 0, 1, 0, 1), (0, 0, 0, 0), (1, 0, 0, 0, 1, 1)])
def test_both_warps_of_a_pair_take_the_same_items(has_chunk):
    items = tuple(i for i, c in enumerate(has_chunk) if c)
    assert outcomes(has_chunk, claim_words()) == {(items, items)}
