"""Counters that several CTAs of a group (or warps of a CTA) add to and then
branch on: under every schedule of the accesses around the barriers, all of
them have to read the same counts, or some leave a loop that the others wait
in. The accesses are taken from the kernel's source in program order and run
through every interleaving of two participants."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_20286_gb300", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _block(text, start):
    """From `start` to the brace that closes the first one opened after it."""
    at = text.index(start)
    depth, i = 0, text.index("{", at)
    for j in range(i, len(text)):
        depth += (text[j] == "{") - (text[j] == "}")
        if depth == 0:
            return text[at:j + 1]
    raise ValueError(start)


def _accesses(text, word, barrier):
    """(kind, slot expression) of the accesses to `word` and the barriers, in
    program order; the slot expression is "" for a plain counter."""
    sub = r"(?:\[([^\]]*)\])?"
    kinds = [("barrier", barrier + "()"), ("read", r"(?:ld_volatile\(&|=\s*)(?:\w+(?:\.|->))*" + word + sub),
             ("add", r"(?:atomicAdd\(&|append\([^;]*?&)(?:\w+(?:\.|->))*" + word + sub),
             ("clear", word + sub + r"\s*=\s*0")]
    found = []
    for kind, pattern in kinds:
        found += [(m.start(), kind, m.group(1) or "") for m in re.finditer(pattern, text)]
    return [(kind, slot) for _, kind, slot in sorted(found)]


def _slot(expr, k):
    """Slot of iteration k: front_slot(e) is e % 3, a plain counter slot 0."""
    expr = re.sub(r"front_slot", "", expr).replace("k_front", "k")
    return eval(expr, {"k": k}) % 3 if expr else 0


def _schedules(programs):
    """Sequences of counts that the participants read, over every schedule.
    programs: per participant a list of (kind, slot, amount)."""
    n = len(programs)
    start = ((0,) * n, (0,) * n, (0, 0, 0), ((),) * n)  # positions, barriers reached, slots, reads
    seen, todo, ends = {start}, [start], set()
    while todo:
        pos, epoch, slots, reads = todo.pop()
        moved = False
        for i, prog in enumerate(programs):
            if pos[i] == len(prog):
                continue
            kind, slot, amount = prog[pos[i]]
            e, s, r = list(epoch), list(slots), list(reads)
            if kind == "wait":
                if min(epoch) < epoch[i]:
                    continue
            elif kind == "arrive":
                e[i] += 1
            elif kind == "read":
                r[i] += (slots[slot],)
            elif kind == "add":
                s[slot] += amount
            else:
                s[slot] = 0
            moved = True
            nxt = (pos[:i] + (pos[i] + 1,) + pos[i + 1:], tuple(e), tuple(s), tuple(r))
            if nxt not in seen:
                seen.add(nxt)
                todo.append(nxt)
        if not moved:
            ends.add(reads)
    return ends


def _reads(before, loop, rounds=5):
    """The counts that both participants read in `before` and `rounds` passes of
    `loop`, None when they depend on the schedule or on the participant."""
    programs = []
    for rank in range(2):
        prog = []
        for k, ops in [(0, before)] + [(k, loop) for k in range(rounds)]:
            for kind, expr in ops:
                if kind == "barrier":
                    prog += [("arrive", 0, 0), ("wait", 0, 0)]
                elif kind != "clear" or rank == 0:  # the first one clears
                    prog.append((kind, _slot(expr, k), 1 + 2 * rank + 10 * k))
        programs.append(prog)
    ends = _schedules(programs)
    return next(iter(ends))[0] if len(ends) == 1 and len(set(next(iter(ends)))) == 1 else None


def _added(k):  # by both participants in iteration k
    return sum(1 + 2 * rank + 10 * k for rank in range(2))


def test_the_check_itself():
    add, read, bar = ("add", ""), ("read", ""), ("barrier", "")
    assert _reads([], [read, add, bar]) is None      # a total read while others add to it
    assert _reads([], [add, bar, read]) is None
    assert _reads([], [add, bar, read, bar], 3) == (4, 28, 72)


def test_front_counts_of_the_tree():
    ops = _accesses(_block(_source("k_fronts.cu"), "for (;; ++k_front)"), "(?:ranked|front_new)", "group_sync")
    assert [k for k, _ in ops].count("read") == 1 and [k for k, _ in ops].count("add") == 1
    assert _reads([], ops) == (0,) + tuple(_added(k) for k in range(4))  # the front before


def test_front_counts_of_the_matrix():
    text = _block(_source("k_peel.cu"), "k_peel(Plan* plan)")
    loop = _block(text, "while (total < target)")
    first, ops = (_accesses(t, "(?:ranked|front_new)", "group_sync") for t in (text[:text.index(loop)], loop))
    assert [k for k, _ in first] == ["add", "barrier", "read"]
    assert [k for k, _ in ops].count("read") == 1 and [k for k, _ in ops].count("add") == 1
    assert _reads(first, ops) == (_added(0),) + tuple(_added(k) for k in range(5))


def test_near_points_of_a_tile():
    """The way from tile to tile of k_igd_near that adds to the list only."""
    loop = _block(_block(_source("k_generation.cu"), "k_igd_near(const float*"), "for (int64_t i0 =")
    ops = _accesses(loop[:loop.index("continue;")], "s_near_n", "__syncthreads")
    assert [k for k, _ in ops][:3] == ["add", "barrier", "read"]
    assert _reads([], ops) == tuple(sum(_added(q) for q in range(k + 1)) for k in range(5))
