"""Model of Finalize's one-launch plan (host logic, no GPU).

An entry packs a window of the chain from its position on, next | min << 16 in
the low word and dist | len << 16 in the high one: where the window ends, its
least position + 1 (0: the path's free end), the distance to that one and the
window's length.  Every step joins each window with the one at its end, in place, so
an entry is read while its owner rewrites it.  The model replays the steps with
reads that see the neighbour before or after its own update (random order, or
as it was when the step began) and checks heads and ranks against the chains
walked directly.  With reads that may take one word from before the update and
one from after it the result is wrong: the 64-bit accesses have to be whole,
which for another CTA's shared memory only relaxed (or stronger) accesses are.
"""
import os
import random
import re

import pytest
from test_jump_model import random_map

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_05302_gb300", "csrc")
FZ_LEN = 0xFFFE


def plan(succ, n, rng, schedule):
    e = [(succ[x], x + 1, 0, 1) if x in succ else (x, 0, 0, 0) for x in range(n)]
    for _ in range(34):
        before, more = list(e), False
        order = list(range(n))
        rng.shuffle(order)
        for x in order:
            nxt, mn, dist, ln = e[x]
            if mn == 0 or ln >= n:
                continue
            old, new = before[nxt], e[nxt]
            f = old if schedule == "step" or (schedule == "mixed" and rng.random() < 0.5) else new
            if schedule == "torn":
                f = rng.choice((old, new, old[:2] + new[2:], new[:2] + old[2:]))
            if f[1] < mn:
                mn, dist = f[1], ln + f[2]
            ln = min(ln + f[3], FZ_LEN)
            e[x] = (f[0], mn, dist, ln)
            more |= mn != 0 and ln < n
        if not more:
            return e
    return None


def wrong(e, succ, n):
    """Positions whose head or rank differs from the chain walked directly."""
    if e is None:
        return n
    bad = 0
    for x in succ:
        seen, y = [x], succ[x]
        while y in succ and y != x:
            seen.append(y)
            y = succ[y]
        if y == x:
            m = min(seen)
            bad += (e[x][1], e[x][2]) != (m + 1, seen.index(m))
        else:
            bad += (e[x][0], e[x][1], e[x][2]) != (y, 0, len(seen))
    return bad


@pytest.mark.parametrize("schedule", ["inplace", "step", "mixed"])
@pytest.mark.parametrize("seed", range(4))
def test_heads_and_ranks(seed, schedule):
    rng = random.Random(seed)
    n = rng.choice((1000, 2500, 4097))
    succ = random_map(n, rng)
    assert wrong(plan(succ, n, rng, schedule), succ, n) == 0


def test_one_cycle_through_every_position():
    rng = random.Random(5)
    for n in (2, 3, 64, 65, 2048):
        perm = list(range(n))
        rng.shuffle(perm)
        succ = {a: b for a, b in zip(perm, perm[1:] + perm[:1])}
        assert wrong(plan(succ, n, rng, "step"), succ, n) == 0


def test_halves_of_two_states_are_wrong():
    rng = random.Random(1)
    succ = random_map(3000, rng)
    assert wrong(plan(succ, 3000, rng, "torn"), succ, 3000) > 0


def test_entries_of_other_ctas_are_read_and_written_whole():
    """The source uses relaxed accesses of cluster scope for the entries: of a
    weak access that races with another the memory model promises nothing."""
    common = open(os.path.join(CSRC, "rs_common.cuh")).read()
    body = open(os.path.join(CSRC, "rs_finalize.cu")).read()
    body = body[body.index("void fz_plan("):body.index("k_fz_plan_one(FinArgs")]
    weak = re.findall(r"(\w+)\(uint32_t addr[^)]*\)\s*\{[^}]*?\b(?:ld|st)\.shared::cluster\.u64", common)
    for name in weak:
        # (a 64-bit entry through a weak access; 32-bit flags go across barriers)
        assert not re.search(name + r"\(at\(", body), name
    get = re.search(r"auto get = .*?MULTI \? (\w+)\(at\(x\)\)", body).group(1)
    put = re.search(r"auto put = .*?if \(MULTI\)\s*(\w+)\(at\(x\), e\)", body, re.S).group(1)
    for name, op in ((get, "ld"), (put, "st")):
        fn = re.search(name + r"\(uint32_t addr[^)]*\)\s*\{[^}]*\}", common).group(0)
        assert op + ".relaxed.cluster.shared::cluster.u64" in fn
