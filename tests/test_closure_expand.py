"""The device closure search restated on the CPU: one launch per level, in
which warps take the members of that level from a list that the same launch
appends to (tag a dependency, reserve a slot, write it: three steps that other
warps' steps may come between). Under any interleaving a warp may only read
list slots that were written before, and the members must be the closure.

With the number of members read from the word that the launch itself raises,
some interleavings read a slot that is reserved and not yet written, whatever
that slot holds: the restatement has to find them, or it would show nothing.
"""
import random

import pytest


class UnwrittenSlot(Exception):
    pass


def graph(rng, n, width):
    deps = [sorted(rng.sample(range(s), rng.randint(0, min(s, width)))) for s in range(n)]
    level = []
    for s in range(n):
        level.append(1 + max((level[d] for d in deps[s]), default=-1))
    return deps, level


def walk(deps, seeds):
    seen, stack = set(seeds), list(seeds)
    while stack:
        for d in deps[stack.pop()]:
            if d not in seen:
                seen.add(d)
                stack.append(d)
    return seen


def search(rng, deps, level, seeds, warps, settled):
    """The members found; settled: the bound of a level's launch is the sum of
    what the seeds and the earlier launches added, else the running total."""
    n_seg, top = len(deps), max(level[s] for s in seeds)
    lst, mark = [None] * n_seg, [False] * n_seg
    found = [0] * (top + 2)
    for i, s in enumerate(seeds):
        lst[i], mark[s] = s, True
    found[top + 1] = len(seeds)

    def warp(w, lv):
        bound = sum(found[lv + 1:]) if settled else sum(found)
        before = sum(found[lv + 1:])
        yield
        for i in range(w, bound, warps):
            s = lst[i]
            if s is None:
                raise UnwrittenSlot
            yield
            if level[s] != lv:
                continue
            for k in range(0, len(deps[s]), 4):  # (a warp of four lanes)
                fresh = []
                for d in deps[s][k:k + 4]:
                    if not mark[d]:
                        mark[d] = True
                        fresh.append(d)
                    yield
                at = before + found[lv]
                found[lv] += len(fresh)
                yield
                for j, d in enumerate(fresh):
                    assert lst[at + j] is None
                    lst[at + j] = d
                    yield

    for lv in range(top, 0, -1):
        running = [warp(w, lv) for w in range(warps)]
        while running:
            w = rng.choice(running)
            for _ in range(rng.choice((1, 1, 2, 8, 40))):  # (bursts: warps that start late)
                if next(w, "done") == "done":
                    running.remove(w)
                    break
    members = lst[:sum(found)]
    assert None not in members and len(set(members)) == len(members)
    return set(members)


@pytest.mark.parametrize("seed", range(60))
def test_members_under_any_interleaving(seed):
    rng = random.Random(seed)
    deps, level = graph(rng, rng.randint(2, 90), rng.randint(1, 12))
    lo = rng.randrange(len(deps))
    seeds = list(range(lo, min(len(deps), lo + rng.randint(1, 5))))
    for warps in (1, 3, 8):
        assert search(rng, deps, level, seeds, warps, settled=True) == walk(deps, seeds)


def test_running_total_reads_unwritten_slots():
    hits = 0
    for seed in range(60):
        rng = random.Random(seed)
        deps, level = graph(rng, 90, 12)
        try:
            search(rng, deps, level, [89], 8, settled=False)
        except UnwrittenSlot:
            hits += 1
    assert hits
