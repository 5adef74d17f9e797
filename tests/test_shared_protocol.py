"""The hand-over between the three teams of the shared kernel
(csrc/mk_bootstrap_shared.cuh), as a model run under random interleavings:
named barriers, mbarriers of the matrix products and their TMEM columns.

Checked for every party count, random skipped steps, two gates a CTA:
  * every team reads from TMEM the products of the gate, step and polynomial
    it is at, and team 0 the shares of that step; no columns are written while
    they are being read, and no team has two products under way;
  * nothing deadlocks, nobody arrives twice at a named barrier;
  * if a wait for products runs out (all later ones then return at once), the
    teams still pass every barrier in order, and no product is in flight when
    TMEM is freed.
Planted mistakes are caught: team 1 arriving at barrier 6 without waiting
there (it can then arrive at barrier 4 twice), and an exit that does not wait
for the products."""
import random

import pytest


def others_of(k):
    m = k - 1
    c2 = min((k + 3) // 3, m)
    c0 = (m - c2 + 1) // 2
    return [0, c0, m - c2], [c0, m - c2 - c0, c2]


class Named:
    def __init__(self, need):
        self.need, self.arrived, self.gen = need, [], 0

    def arrive(self, who):
        assert who not in self.arrived, "double arrival"
        self.arrived.append(who)
        if len(self.arrived) == self.need:
            self.arrived, self.gen = [], self.gen + 1


def run_cta(k, n, steps, seed, runs_out=False, mutant=None):
    rnd = random.Random(seed)
    out_at = rnd.randrange(1, 200) if runs_out else None
    first, count = others_of(k)
    named = {0: Named(3), 4: Named(3), 6: Named(2), 7: Named(2), 9: Named(3)}
    phases = [0] * 4             # completed phases of the mbarriers: the teams', v's
    flight = []                  # (mbarrier, products, columns), by team of issue: columns
    tmem, shares = [None] * 3, [None] * 3
    limit = k * n

    def next_step(s):
        while s < limit and not steps[s]:
            s += 1
        return s

    def team(t):
        mine = count[t]
        slots, phase, vphase = mine + (t < 2), 0, 0
        for gate in range(2):
            reading = started = False
            party, step = 1, next_step(0)
            while step < limit:
                i, nxt = step // n + 1, next_step(step + 1)
                if i != party:
                    yield ("sync", 9)
                    party = i

                def poly(s):
                    if s == mine:
                        return i if t else 0
                    o = first[t] + s + 1
                    return o if o < i else o + 1
                if not started:
                    yield ("issue", t, t, (gate, step, poly(0)))
                started = slots > 1 and nxt < limit and nxt // n + 1 == i
                for s in range(slots + (t < 2)):
                    last = s == slots
                    if last:
                        yield ("wait", 3, vphase)
                        vphase += 1
                    else:
                        yield ("wait", t, phase)
                        phase += 1
                    at = (0, (gate, step, "v")) if last else (t, (gate, step, poly(s)))
                    yield ("holds",) + at
                    yield ("holds",) + at  # still, at the end of the read
                    if last:
                        yield ("arrive" if mutant == "arrive_at_6" and t == 1 else "sync", 6)
                    if s + 1 < slots:
                        yield ("issue", t, t, (gate, step, poly(s + 1)))
                    elif started and last == (t == 0):
                        yield ("issue", t, t, (gate, nxt, poly(0)))
                    if s == slots - 1 and t:
                        if t == 2 and reading:
                            yield ("sync", 7)
                        yield ("share", t, (gate, step))
                        yield ("arrive", 4)
                        reading = True
                    elif s == slots - 1:
                        yield ("sync", 4)
                        yield ("shared", (gate, step))
                        yield ("shared", (gate, step))
                        yield ("arrive", 7)
                        yield ("issue", 3, 0, (gate, step, "v"))
                step = nxt
            if t == 2 and reading:
                yield ("sync", 7)
            yield ("sync", 0)
        if mutant != "no_drain":
            yield ("drain", t)
        yield ("sync", 0)
        yield ("freed",)

    gens = [team(t) for t in range(3)]
    op = [next(g) for g in gens]
    clock = 0

    def ready(t):
        o = op[t]
        if o is None:
            return False
        if o[0] == "wait":
            return (runs_out and clock >= out_at) or (phases[o[1]] & 1) != (o[2] & 1)
        if o[0] == "blocked":
            return named[o[1]].gen != o[2]
        return o[0] != "drain" or all(columns != o[1] for _, _, columns in flight)

    while any(o is not None for o in op):
        moves = [t for t in range(3) if ready(t)] + (["product"] if flight else [])
        assert moves, "deadlock"
        m = rnd.choice(moves)
        clock += 1
        if m == "product":
            bar, what, columns = flight.pop(rnd.randrange(len(flight)))
            tmem[columns] = what
            phases[bar] += 1
            continue
        o = op[m]
        if o[0] == "sync":
            op[m] = ("blocked", o[1], named[o[1]].gen)
            named[o[1]].arrive(m)
            continue
        if o[0] == "arrive":
            named[o[1]].arrive(m)
        elif o[0] == "issue":
            assert runs_out or all(columns != o[2] for _, _, columns in flight), "two products under way"
            tmem[o[2]] = None
            flight.append((o[1], o[3], o[2]))
        elif o[0] == "share":
            shares[o[1]] = o[2]
        elif o[0] == "holds":
            assert runs_out or tmem[o[1]] == o[2], "other products in the columns"
        elif o[0] == "shared":
            assert runs_out or shares[1:] == [o[1]] * 2, "shares of another step"
        elif o[0] == "freed":
            assert not flight, "in flight when TMEM is freed"
        op[m] = next(gens[m], None)
    assert all(not b.arrived for b in named.values())


def cases(k, runs):
    for seed in range(runs):
        r = random.Random(seed)
        n, share = r.choice([1, 2, 3, 5]), r.choice([0.3, 0.9, 1])
        yield n, [r.random() < share for _ in range(k * n)], seed


@pytest.mark.parametrize("runs_out", [False, True])
@pytest.mark.parametrize("k", range(2, 9))
def test_hand_over(k, runs_out):
    for n, steps, seed in cases(k, 120):
        run_cta(k, n, steps, seed, runs_out)


@pytest.mark.parametrize("mutant,says", [("arrive_at_6", "double arrival"), ("no_drain", "in flight")])
def test_planted_mistakes_are_caught(mutant, says):
    caught = 0
    for k in range(2, 9):
        for n, steps, seed in cases(k, 120):
            try:
                run_cta(k, n, steps, seed, True, mutant)
            except AssertionError as e:
                caught += says in str(e)
    assert caught
