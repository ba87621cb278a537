"""The named barriers of the pair scan (csrc/fwd_pair.cu) on the CPU: every
interleaving of a CTA's warps over a few chunks, as far as its barriers and the
products' completions order them.  A barrier that a warp arrives at again before
all its threads have joined the time before counts that warp for another one,
and what it orders comes apart, or it never completes.  The program below is the
kernel's, two of the element-wise warps for the sixteen; which barrier stands
before the last chunk's results is read from the source."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2509_25223_gb300", "csrc", "fwd_pair.cu")


def _tail_barriers():
    """The barriers (ids) that the copying and the element-wise warps join behind
    the loop, before the last chunk's results, and the id of kBarO."""
    text = open(SRC).read()
    ids = {n: int(v) for n, v in re.findall(r"\b(kBar[A-Z])\s*=\s*(\d+)", text)}
    assert len(set(ids.values())) == len(ids) and 0 not in ids.values()
    tails = [text[m.end():m.end() + 400] for m in re.finditer(r"if \(alive && NC > 0\) \{", text)]
    names = [re.search(r"bar_sync\((kBar[A-Z]), kHandThreads\)", t).group(1) for t in tails]
    assert len(names) == 2
    return [ids[n] for n in names], ids["kBarO"]


def _programs(NC, rdn, tail_copy, tail_elem, O):
    """Per role a list of (operation, object): sync / arrive on a barrier, wait for
    an event, set one."""
    X, E, ALL = "X", "E", "all"
    issue, copy, elem = [], [("set", ("A", 0)), ("set", ("B", 0))], []
    for c in range(NC):
        issue += [("sync", ALL), ("set", ("mma1", c))]
        copy += [("sync", ALL)]
        elem += [("sync", ALL)]
        if rdn:
            issue += [("sync", X), ("wait", ("A", c)), ("set", ("mma2", c))]
        issue += [("sync", E), ("set", ("mma4", c)), ("wait", ("B", c)), ("set", ("mma3", c))]
        if c:
            copy += [("wait", ("mma3", c - 1)), ("set", ("B", c)), ("sync", O)]
            elem += [("wait", ("mma3", c - 1)), ("arrive", O)]
        if rdn:
            copy += [("wait", ("mma2", c)), ("set", ("A", c + 1))]
        copy += [("wait", ("mma4", c))]
        elem += [("wait", ("mma1", c))]
        if rdn:
            elem += [("arrive", X), ("wait", ("mma2", c))]
        elem += [("arrive", E), ("wait", ("mma4", c))]
    issue += [("sync", ALL)]
    copy += [("sync", tail_copy), ("sync", O), ("sync", ALL)]
    elem += [("sync", tail_elem), ("wait", ("mma3", NC - 1)), ("arrive", O), ("sync", ALL)]
    return [issue, copy, elem, elem]


def _explore(progs, members):
    """Every reachable state: asserts that no warp arrives twice within one use of
    a barrier and that every warp ends."""
    start = (tuple(0 for _ in progs), frozenset(), frozenset())  # next op, joined, events
    seen, todo = {start}, [start]
    while todo:
        pcs, joined, events = todo.pop()
        moved = False
        for r, pc in enumerate(pcs):
            if pc == len(progs[r]):
                continue
            op, what = progs[r][pc]
            blocked = op == "sync" and (r, what) in joined
            if blocked or (op == "wait" and what not in events):
                continue
            nj, ne, npc = joined, events, list(pcs)
            if op in ("sync", "arrive"):
                assert (r, what) not in joined, f"warp {r} arrives at barrier {what} twice"
                nj = joined | {(r, what)}
                if op == "arrive":
                    npc[r] += 1
                if all((m, what) in nj for m in members[what]):  # complete: all go on
                    nj = frozenset(x for x in nj if x[1] != what)
                    for m in members[what]:
                        if npc[m] < len(progs[m]) and progs[m][npc[m]] == ("sync", what):
                            npc[m] += 1
            else:
                npc[r] += 1
                if op == "set":
                    ne = events | {what}
            state = (tuple(npc), nj, ne)
            moved = True
            if state not in seen:
                seen.add(state)
                todo.append(state)
        assert moved or all(pc == len(p) for pc, p in zip(pcs, progs)), "a warp waits for ever"


@pytest.mark.parametrize("rdn", [True, False])
@pytest.mark.parametrize("NC", [1, 2, 4])
def test_no_barrier_is_arrived_at_again_before_it_completes(NC, rdn):
    (tail_copy, tail_elem), O = _tail_barriers()
    members = {"all": [0, 1, 2, 3], "X": [0, 2, 3], "E": [0, 2, 3]}
    for b in {tail_copy, tail_elem, O}:
        members[b] = [1, 2, 3]
    _explore(_programs(NC, rdn, tail_copy, tail_elem, O), members)


def test_the_hand_over_is_taken_after_its_values_are_used():
    """CTA 1 tells CTA 0 that the hand-over buffer may be written again by an
    arrival that orders no earlier load: it has to stand behind the use of
    everything read from there, r as well as ob, in either method."""
    text = open(SRC).read()
    part = text[text.index("float r[16], ob[16];"):text.index("publish(kBarE);", text.index("float r[16], ob[16];"))]
    taken = [m.start() for m in re.finditer(r"taken\(got\);", part)]
    assert len(taken) == 2
    rdn_use, rla_use = part.index("r[i] - gm[i] * x[i]"), part.index("e[i] = r[i]")
    puts = [m.start() for m in re.finditer(r"tmem_st16\(tm \+ lane \+ T_D1 \+ 64 \+ g16, ob\)", part)]
    assert rdn_use < puts[0] < taken[0] and max(rla_use, puts[1]) < taken[1]
