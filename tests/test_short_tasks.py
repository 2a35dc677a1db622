"""The waits by parity between the thread that posts tasks and copies tiles and the one that issues MMAs in the scorer of one
short layer (csrc/score_short.cuh), on the CPU: every interleaving of the two, of the copies' arrivals and of the
commits', for the tasks a CTA may draw.  A wait on a phase lets through whoever is two phases early, so that tiles are taken
before they are there, and holds whoever comes two phases late for good."""
import itertools

import pytest

K0, K1, Q0, Q1 = range(4)


def tasks_of(drawn, posts_empty=False):
    """What a CTA posts that drew `drawn`, each (barriers of pass 1, barriers of pass 2 in the order of its waits)."""
    posted, loaded = [], None
    for own, pass_ in [(i, 0) for i in range(len(drawn))] + [(i, 1) for i in reversed(range(len(drawn)))]:
        waits = drawn[own][pass_]
        if waits or posts_empty:
            posted.append((pass_, waits, own != loaded))
            if own != loaded:
                loaded = own
    return posted


def programs(posted):
    """Steps of the producer and of the MMA warp.  wait: (barrier, phase); copies and commits arrive later."""
    producer, mma, loads = [], [], 0
    for n, (pass_, waits, fresh) in enumerate(posted):
        producer += [("wait", ("empty", n % 2), n // 2 - 1), ("arrive", ("full", n % 2))]
        mma += [("wait", ("full", n % 2), n // 2), ("arrive", ("empty", n % 2))]
        if fresh:
            if n:
                producer.append(("wait", "done", n - 1))
            if loads:
                producer += [("wait", b, loads - 1) for b in range(4)]
            producer.append(("copy", n))
            loads += 1
        mma += [("take", b, loads - 1) for b in waits] + [("commit",)]
        if pass_ == 0:
            producer.append(("wait", "done", n))
    return producer, mma


def faults(posted):
    """Of all interleavings: "early" products, copies over tiles that are in use, and ends where nobody can go on."""
    producer, mma = programs(posted)
    names = ["done", ("full", 0), ("full", 1), ("empty", 0), ("empty", 1), 0, 1, 2, 3]
    at = {x: i for i, x in enumerate(names)}
    found, seen, todo = set(), set(), [((0, 0), (0,) * len(names), (0,) * 4, 0)]

    def add(t, i):
        return t[:i] + (t[i] + 1,) + t[i + 1:]

    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        pc, phases, issued, commits = state
        passes = lambda name, phase: phase < 0 or phases[at[name]] % 2 != phase % 2
        before = len(todo)
        for who, program in enumerate((producer, mma)):
            if pc[who] == len(program):
                continue
            step, moved = program[pc[who]], add(pc, who)
            if step[0] == "arrive":
                todo.append((moved, add(phases, at[step[1]]), issued, commits))
            elif step[0] == "commit":
                todo.append((moved, phases, issued, commits + 1))
            elif step[0] == "copy":
                if phases[at["done"]] < step[1]:
                    found.add("tiles in use")
                todo.append((moved, phases, tuple(i + 1 for i in issued), commits))
            elif passes(step[1], step[2]):
                if step[0] == "take" and phases[at[step[1]]] <= step[2]:
                    found.add("early")
                todo.append((moved, phases, issued, commits))
        for b in range(4):
            if phases[at[b]] < issued[b]:
                todo.append((pc, add(phases, at[b]), issued, commits))
        if phases[at["done"]] < commits:
            todo.append((pc, add(phases, at["done"]), issued, commits))
        if len(todo) == before and pc != (len(producer), len(mma)):
            found.add("stall")
    return found


# (pass 1, pass 2): a segment's first half and its second, with and without a tile of its own; whole segments of one pair of tiles, of
# half a row block, of two pairs
FIRST, SECOND, EMPTY = ([K0, Q0], [K0, Q0, Q1]), ([K0, Q1], [K0, Q0, Q1]), ([K0, Q1], [])
WHOLE, HALF_BLOCK, TWO = ([K0, Q0, Q1], [K0, Q0, Q1]), ([K0, Q0], [K0, Q0, Q1]), ([K0, Q0, Q1, K1], [K0, Q0, Q1, K1])


@pytest.mark.parametrize("kinds", [(FIRST, SECOND, EMPTY), (WHOLE, TWO), (HALF_BLOCK, TWO)])
@pytest.mark.parametrize("n", [1, 2, 3])
def test_every_wait_is_for_its_own_phase(kinds, n):
    for drawn in itertools.product(kinds, repeat=n):
        assert not faults(tasks_of(drawn)), drawn


def test_what_posting_second_passes_without_a_tile_does():
    assert faults(tasks_of((EMPTY, FIRST), posts_empty=True)) == {"stall"}
    assert "early" in faults(tasks_of((FIRST, EMPTY, FIRST), posts_empty=True))
