"""How long a slot of the resident scorer's tagged words lives, on the CPU: CTAs of a team as counters of the units they have
been through, with the waits of csrc/score_res.cuh and the sizes its headers state (`ahead`: teams whose rows have common
references, found so many units before).  One step of one CTA is held back while
all others go as far as their waits let them; whatever it has still to read must not have been written over."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_06746_b200", "csrc")
STEPS = ("statistics", "published", "known", "entropies", "summed")


def constant(header, name):
    with open(os.path.join(CSRC, header)) as f:
        return int(re.search(rf"constexpr int {name} = (\d+);", f.read()).group(1))


def found(done, ahead):
    """References are there of the first `ahead` units, then of unit u + ahead once the CTA whose turn it is has published u."""
    u = ahead
    while done[u % len(done)]["published"] > u - ahead:
        u += 1
    return u


def run(ring, units, ctas=41, held=None, ahead=None):
    """Units every CTA has been through, per step, once nothing moves; `held` = (CTA, step, unit) never happens."""
    done = [dict.fromkeys(STEPS, 0) for _ in range(ctas)]

    def may(c, step):
        d = done[c]
        u = d[step]
        if u == units or held == (c, step, u):
            return False
        if ahead is not None and step in ("statistics", "published", "known") and found(done, ahead) <= u:
            return False
        return {"statistics": d["summed"] + ring > u,                 # a place for the unit's statistics
                "published": d["statistics"] > u,
                # one warp: it knows a unit once all CTAs have published it, leaves its entropies, then goes on
                "known": d["entropies"] == u and all(o["published"] > u for o in done),
                "entropies": d["known"] > u,
                "summed": d["known"] > u}[step]

    moved = True
    while moved:
        moved = False
        for c in range(ctas):
            for step in STEPS:
                while may(c, step):
                    done[c][step] += 1
                    moved = True
    return done


def test_nobody_waits_for_good():
    ring = constant("score_res.cuh", "kResRing")
    for ahead in (None, 2 * ring):
        assert all(set(d.values()) == {5 * ring} for d in run(ring, 5 * ring, ahead=ahead))


@pytest.mark.parametrize("step", ["known", "entropies"])
def test_words_outlive_their_last_reader(step):
    ring, slots = constant("score_res.cuh", "kResRing"), constant("common.cuh", "kXchSlots")
    for unit in range(2 * ring + 2):
        done = run(ring, 8 * ring, ctas=3, held=(0, step, unit))
        latest = max(d["published"] for d in done) - 1
        assert latest < unit + slots, f"unit {latest} is written over unit {unit} while {step} reads it"


@pytest.mark.parametrize("step", ["statistics", "published", "known"])
def test_references_outlive_their_last_reader(step):
    ring, slots = constant("score_res.cuh", "kResRing"), constant("common.cuh", "kRefSlots")
    for unit in range(0, 2 * ring + 2, 3):
        done = run(ring, 8 * ring, held=(0, step, unit), ahead=2 * ring)
        latest = found(done, 2 * ring) - 1
        assert latest < unit + slots, f"unit {latest} is written over unit {unit} while {step} reads it"
