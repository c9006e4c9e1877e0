"""The named barriers of a team of attn_i8_kernel, on which some warps only arrive: their phases must stay apart by the order of
the warps' own steps.  The waits in between cannot be relied on for it: they give up when one of them runs out, and the kernel
has to end all the same.  Played through on the host, with waits that hold nothing up, over many orders of the warps' steps;
the barrier ids are read from the source."""
import os
import random
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_01831_b200", "csrc")


def _team_barriers():
    """The ids of a team's barriers, from the source."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "attention_i8.cuh")).read())
    decl = re.search(r"const int (bar_tm = [^;]+);", text).group(1)
    ids = {}
    for part in decl.split(","):
        name, expr = part.split("=")
        ids[name.strip()] = expr.strip()
    return {n: (lambda tm, e=e: eval(e, {"tm": tm})) for n, e in ids.items()}, text


class _Stuck(Exception):
    pass


def _play(ids, warps, units, rng):
    """One order of the steps of a team's warps over `units` units in which no wait holds anything up.  A warp that is not the
    issuing one only arrives where the K levels and where the weights are complete; all synchronise at the question whether to
    restart.  Returns the (unit, step) pairs that met in one phase of a barrier, per phase."""
    def program(w):
        for u in range(units):
            yield ("sync" if w == 0 else "arrive", ids["k"], (u, "k"))
            yield ("sync", ids["tm"], (u, "vote"))
            yield ("sync" if w == 0 else "arrive", ids["p"], (u, "p"))
        yield ("sync", ids["tm"], (units, "end"))
    progs = [program(w) for w in range(warps)]
    todo = [next(p) for p in progs]
    count, phases, members, blocked = {}, {}, {}, [False] * warps
    while any(t is not None for t in todo):
        ready = [w for w in range(warps) if todo[w] is not None and not blocked[w]]
        if not ready:
            raise _Stuck
        w = rng.choice(ready)
        kind, bar, what = todo[w]
        members.setdefault(bar, []).append(what)
        count[bar] = count.get(bar, 0) + 1
        waiting = [v for v in range(warps) if blocked[v] and todo[v][1] == bar]
        if kind == "sync":
            blocked[w] = True
            waiting.append(w)
        else:
            todo[w] = next(progs[w], None)
        if count[bar] == warps:
            phases.setdefault(bar, []).append(set(members[bar]))
            count[bar], members[bar] = 0, []
            for v in waiting:
                blocked[v] = False
                todo[v] = next(progs[v], None)
    return phases


def _mixed(ids, warps=4, units=6, orders=400):
    bad = 0
    for seed in range(orders):
        try:
            phases = _play(ids, warps, units, random.Random(seed))
        except _Stuck:
            bad += 1
            continue
        bad += any(len(s) > 1 for ps in phases.values() for s in ps)
    return bad


def test_phases_of_the_teams_barriers_never_mix():
    ids, text = _team_barriers()
    used = {n: re.search(r"bar_arrive\(%s," % n, text) is not None for n in ids}
    arrives = [n for n in ids if used[n]]
    assert len(arrives) == 2 and "bar_k" in arrives, "the steps played below are the kernel's"
    p = [n for n in arrives if n != "bar_k"][0]
    for tm in range(4):
        assert _mixed({"k": ids["bar_k"](tm), "tm": ids["bar_tm"](tm), "p": ids[p](tm)}) == 0


def test_a_shared_barrier_would_mix():
    assert _mixed({"k": 10, "tm": 1, "p": 1}) > 0


def test_barrier_ids_are_distinct():
    ids, text = _team_barriers()
    fixed = [int(x) for x in re.findall(r"named_bar\((\d+), (?:T \* TT|C::kThreads)\)", text)]
    assert len(fixed) == 2
    every = [0] + fixed + [f(tm) for f in ids.values() for tm in range(4)]
    assert len(set(every)) == len(every) and max(every) < 16


def _decisions(flag_of, warps=4, units=8, orders=400):
    """Units in which a team's warps do not agree whether to restart, over many orders of their steps: a warp may raise the unit's flag,
    all meet, each looks at the flag, and a team that restarts meets twice more with the flag taken back in between."""
    split = 0
    for seed in range(orders):
        rng, flags, seen = random.Random(seed), {}, [dict() for _ in range(warps)]

        def program(w):
            for u in range(units):
                if rng.random() < 0.1:
                    flags[flag_of(u)] = 1
                    yield "step"
                yield "sync"
                seen[w][u] = flags.get(flag_of(u), 0)
                yield "step"
                if seen[w][u]:
                    yield "sync"
                    if w == 0:
                        flags[flag_of(u)] = 0
                    yield "sync"
                    yield "sync"
        progs, waiting, done = [program(w) for w in range(warps)], set(), set()
        while len(done) < warps:
            ready = [w for w in range(warps) if w not in waiting and w not in done]
            if not ready:
                if len(waiting) + len(done) < warps or done:
                    break                       # warps that took different ways wait for one another
                waiting.clear()
                continue
            w = rng.choice(ready)
            step = next(progs[w], None)
            if step is None:
                done.add(w)
            elif step == "sync":
                waiting.add(w)
        split += len(done) < warps or any(len({s.get(u) for s in seen}) > 1 for u in range(units))
    return split


def test_all_warps_take_the_restart_or_none_does():
    """The question is asked at a barrier that gives all threads one answer; a flag in memory would have to be one per unit."""
    assert re.findall(r"([^\n]*)\brestart\(\);", _team_barriers()[1]) == ["        if (bar_or(bar_tm, TT, forced || over)) "]
    assert _decisions(lambda u: u) == 0


def test_one_flag_for_all_units_would_split_the_team():
    assert _decisions(lambda u: 0) > 0
