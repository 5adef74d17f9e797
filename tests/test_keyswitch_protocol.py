"""The mbarrier protocol of the matrix-product key switch
(csrc/mk_keyswitch_tc.cu), as a model run under random interleavings.

Roles of a CTA over its coefficient pairs kb = 0 .. nkb - 1 (stage kb % 4):
  copy warp -- waits empty[stage] for kb >= 4, issues the key tile's bulk copy
               (completes full[stage]); at its end waits for its last copies;
  builders  -- each waits empty[stage] for kb >= 4, writes its indicators,
               arrives on ready[stage]; then waits for `done` and reads TMEM;
  MMA warp  -- waits full[stage] and ready[stage], issues the products,
               commits empty[stage]; at its end commits `done` and waits for it.
Waits between roles may run out at any moment (they are bounded) and then set
the abort word, on which every later wait that is not satisfied gives up; the
waits for a role's own copies and products at its end do not look at it.

Checked: products read the pair they are for; a stage is overwritten only once
the products that read it are done; whatever runs out, no copy and no product
is in flight when the CTA frees its TMEM and leaves.  A planted mistake (the
MMA warp waits for its products only if one of its own waits ran out) is
caught: a builder's wait for `done` can run out after all products are issued.
"""
import random

import pytest

STAGES = 4


class Bar:
    def __init__(self, count):
        self.count, self.pending, self.phase = count, count, 0

    def arrive(self):
        self.pending -= 1
        if self.pending == 0:
            self.pending, self.phase = self.count, self.phase + 1

    def passed(self, parity):
        return (self.phase & 1) != parity


def run_cta(nkb, builders, seed, give_up, mutant=None):
    """give_up: chance that a wait between roles runs out at a look."""
    rnd = random.Random(seed)
    full, empty = [Bar(1) for _ in range(STAGES)], [Bar(1) for _ in range(STAGES)]
    ready, done = [Bar(builders) for _ in range(STAGES)], Bar(1)
    abort, copies, products, tmem = [False], [], [], []
    tile, built = [None] * STAGES, [[None] * builders for _ in range(STAGES)]

    def wait(bar, parity):  # kt_wait with the abort word
        while not bar.passed(parity):
            if abort[0]:
                return False
            if rnd.random() < give_up:
                abort[0] = True
                return False
            yield
        return True

    def own(bar, parity):  # kt_wait without it: the role's own copies or products
        while not bar.passed(parity):
            yield

    def copy_warp():
        kb = 0
        while kb < nkb:
            st = kb % STAGES
            if kb >= STAGES and not (yield from wait(empty[st], (kb // STAGES - 1) & 1)):
                break
            assert all(s != st for s, _ in products if s is not None), "copy into a stage being read"
            copies.append((st, kb))
            kb += 1
            yield
        for q in range(max(kb - STAGES, 0), kb):
            yield from own(full[q % STAGES], (q // STAGES) & 1)

    def mma_warp():
        ok = True
        for kb in range(nkb):
            st, ph = kb % STAGES, (kb // STAGES) & 1
            ok = (yield from wait(full[st], ph)) and (yield from wait(ready[st], ph))
            if not ok:
                break
            products.append((st, kb))
            yield
        products.append((None, "done"))
        if not (mutant == "drain_if_own_wait_ran_out" and ok):
            yield from own(done, 0)

    def builder(b):
        ok = True
        for kb in range(nkb):
            st = kb % STAGES
            if kb >= STAGES and not (yield from wait(empty[st], (kb // STAGES - 1) & 1)):
                ok = False
                break
            assert all(s != st for s, _ in products if s is not None), "indicators into a stage being read"
            built[st][b] = kb
            yield
            ready[st].arrive()
        if ok and (yield from wait(done, 0)) and not abort[0]:
            assert tmem == list(range(nkb))

    roles = [copy_warp(), mma_warp()] + [builder(b) for b in range(builders)]
    for _ in range(200_000):
        moves = roles + (["copy"] if copies else []) + (["product"] if products else [])
        if not roles:
            break
        m = rnd.choice(moves)
        if m == "copy":
            st, kb = copies.pop(rnd.randrange(len(copies)))
            tile[st] = kb
            full[st].arrive()
        elif m == "product":  # in order
            st, kb = products.pop(0)
            if st is None:
                done.arrive()
                continue
            assert tile[st] == kb and built[st] == [kb] * builders, "products of another pair"
            tmem.append(kb)
            empty[st].arrive()
        else:
            try:
                next(m)
            except StopIteration:
                roles.remove(m)
    assert not roles, "a role never ended"
    assert not copies and not products, "in flight at the exit"
    return abort[0]


@pytest.mark.parametrize("nkb", [16, 48])
def test_undisturbed(nkb):
    for seed in range(60):
        assert not run_cta(nkb, 2, seed, 0.0)


def test_waits_that_run_out_leave_nothing_in_flight():
    assert sum(run_cta(16, 2, seed, 0.01) for seed in range(600)) > 200


def test_planted_mistake_is_caught():
    caught = 0
    for seed in range(600):
        try:
            run_cta(16, 2, seed, 0.01, mutant="drain_if_own_wait_ran_out")
        except AssertionError as e:
            caught += "in flight" in str(e)
    assert caught
