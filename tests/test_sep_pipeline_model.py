"""CPU model check of the warp roles of the separable transforms
(k_sep_adjoint in csrc/sep_adjoint.cu, k_sep_forward in csrc/sep_forward.cu).

The roles meet only at mbarriers, and a wait names a phase by its parity: it
is over as soon as the barrier's last completed phase has that parity, and it
never ends if the barrier has gone one phase further in the meantime. The
model plays every warp's waits, arrivals, reads and writes under random
interleavings (each warp with a speed of its own that changes now and then,
copies and MMAs landing late) and checks that

* no interleaving deadlocks: something can run until every role is done;
* operands, accumulators and step records are overwritten only when all
  their readers are past them, and read only when complete.

In further runs one wait runs out, as all do after about a second, and the
others in turn where they depend on it: every role has to end, no copy may go
to a slot that is still in use, and no copy or MMA may be in flight when the
last role ends, for the memory belongs to the next block then.

The numbers of barriers and what listers and adders do after a wait that ran
out are read from the sources. Mistakes planted in the model (four barriers for the
adjoint's MMAs, which the generators' wait can find two phases on; an operand
buffer taken back early; listers and adders that run on) have to be caught.
"""
import pathlib
import random
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2505_08777_gb300" / "csrc"


def constant(name, file):
    return int(re.search(rf"\b{name} = (\d+)", (CSRC / file).read_text()).group(1))


def lister_leaves(file):
    """Whether the lister leaves its loop before it writes a step into a slot whose wait ran out."""
    text = (CSRC / file).read_text()
    text = text[text.index("// --- steps of this CTA"):]
    return re.search(r"sep_wait\(&empty[^;]*;\s*if \(!ok\) break;[^;]*(;[^;]*){0,8}mbar_expect_tx", text) is not None


ADJ_FULL = constant("kAdjFull", "sep_adjoint.cu")
# meetings of the adjoint's adders: all of them are left if the wait ran out
ADDERS = (CSRC / "sep_adjoint.cu").read_text()
ADDERS_LEAVE = ADDERS.count("if (!add_sync()) break;") == len(re.findall(r"\badd_sync\(\)", ADDERS))
ADJ_LEAVES, FWD_LEAVES = lister_leaves("sep_adjoint.cu"), lister_leaves("sep_forward.cu")


class Violation(AssertionError):
    pass


def check(cond, what):
    if not cond:
        raise Violation(what)


class Barrier:
    def __init__(self, count):
        self.count, self.left, self.tx, self.done = count, count, 0, 0

    def arrive(self):
        self.left -= 1
        check(self.left >= 0, "more arrivals than the barrier counts")
        self.turn()

    def turn(self):
        if self.left == 0 and self.tx == 0:
            self.left, self.done = self.count, self.done + 1

    def passed(self, phase):
        """The hardware's test: by the parity of `phase` alone."""
        return (self.done & 1) != (phase & 1)


class Meeting:
    """A named barrier of n warps that also tells whether one of them stops (barrier.red.or)."""

    def __init__(self, n):
        self.n, self.come, self.gen, self.stop = n, 0, 0, {0: False}

    def arrive(self, stop=False):
        gen = self.gen
        self.stop[gen] = self.stop.get(gen, False) or stop
        self.come += 1
        if self.come == self.n:
            self.come, self.gen = 0, self.gen + 1
        return gen

    def met(self, gen):
        return self.gen > gen


class Model:
    """Roles are generators that yield None (a step), (barrier, phase) (a wait: they are sent whether it was
    over before it ran out) or a function (a named barrier). `fails`: one wait runs out, and then those that
    nothing ends any more."""

    def __init__(self, rng, fails=False):
        self.rng, self.fails, self.failed, self.procs, self.later = rng, fails, False, {}, []

    def add(self, name, gen):
        self.procs[name] = [gen, None]

    def queue(self, what, after=None):
        """An asynchronous completion, in order behind `after`."""
        item = [what, after]
        self.later.append(item)
        return item

    def see(self, cond, what):
        """What holds for the values, as long as no wait has run out."""
        check(cond or self.failed, what)

    def resume(self, name, answer):
        g = self.procs[name]
        try:
            g[1] = g[0].send(answer)
        except StopIteration:
            g[1] = "end"

    @staticmethod
    def can(at):
        return at is None or (at[0].passed(at[1]) if isinstance(at, tuple) else at != "end" and at())

    def play(self):
        speed = {n: 10 ** self.rng.uniform(-2, 0) for n in self.procs}
        speed["async"] = 10 ** self.rng.uniform(-2, 0)
        for n in self.procs:
            self.resume(n, None)
        left = self.rng.randint(1, 1200) if self.fails else -1
        while True:
            live = [n for n, g in self.procs.items() if g[1] != "end"]
            ready = [n for n in live if self.can(self.procs[n][1])]
            land = [x for x in self.later if x[1] is None or x[1] not in self.later]
            if not live:
                check(not land, "copies or MMAs in flight at the end")
                return
            waits = [n for n in live if isinstance(self.procs[n][1], tuple) and n not in ready]
            left -= 1
            if waits and (left == 0 or self.failed and not ready and not land):
                self.failed = True
                self.resume(self.rng.choice(waits), False)
                continue
            check(ready or land, "every role waits: " + ", ".join(sorted(live)))
            names = ready + (["async"] if land else [])
            pick = self.rng.choices(names, [speed[n] for n in names])[0]
            if self.rng.random() < 0.02:
                speed[self.rng.choice(list(speed))] = 10 ** self.rng.uniform(-3, 0)
            if pick == "async":
                x = self.rng.choice(land)
                self.later.remove(x)
                x[0]()
            else:
                self.resume(pick, True)


class Adjoint(Model):
    """One CTA: chunks of 2^ls strips, tiles ending after the chunks in `ends`."""

    SLOTS, BUFS, DBUFS = 8, 3, 4

    def __init__(self, rng, chunks, ends, nfull=ADJ_FULL, x_wait=True, w_wait=True, leaves=ADJ_LEAVES,
                 adders_leave=ADDERS_LEAVE, fails=False):
        super().__init__(rng, fails)
        self.nf, self.x_wait, self.w_wait, self.leaves = nfull, x_wait, w_wait, leaves
        self.adders_leave, self.sums, self.flag = adders_leave, [0] * 8, -1
        self.steps = []                      # (chunk, strip, last step that used W's buffer, tile end)
        last = []
        for c, ls in enumerate(chunks):
            used = last[c - self.BUFS] if c >= self.BUFS else -1
            for s in range(1 << ls):
                end = s + 1 == 1 << ls and (c in ends or c + 1 == len(chunks))
                self.steps.append((c, s, used, end))
            last.append(len(self.steps) - 1)
        n = self.n = len(self.steps)
        self.full = [Barrier(1) for _ in range(nfull)]
        self.empty = [Barrier(8) for _ in range(self.SLOTS)]
        self.ready = [Barrier(1) for _ in range(self.SLOTS)]
        self.listed = [Barrier(1) for _ in range(self.SLOTS)]
        self.summed = Barrier(8)
        self.slot = [None] * self.SLOTS      # step whose record it holds
        self.copying = [False] * self.SLOTS
        self.wrote = [0] * n                 # generator warps past a step's operands
        self.issued, self.done = [False] * n, [False] * n
        self.read = [0] * n                  # adder warps done with a step's sums
        self.meet = [Meeting(8), Meeting(8)]
        self.add("lister", self.lister())
        for k in range(3):
            self.add(f"issuer {k}", self.issuer(k))
        for g in range(2):
            for w in range(8):
                self.add(f"generator {g}.{w}", self.generator(g, w))
        for w in range(8):
            self.add(f"adder {w}", self.adder(w))

    def put(self, it, end):
        old = it - self.SLOTS
        if 0 <= old < self.n:
            check(self.read[old] == 8 and self.wrote[old] == 8 and self.issued[old], f"record of step {old} rewritten early")
        check(not self.copying[it % self.SLOTS], "a copy goes to a slot whose last copy is in flight")
        self.slot[it % self.SLOTS] = (it, end)

    def record(self, it):
        check(self.slot[it % self.SLOTS] is not None and self.slot[it % self.SLOTS][0] == it, f"record of step {it} not there")
        return self.slot[it % self.SLOTS][1]

    def lister(self):
        S, ok, it = self.SLOTS, True, 0
        while it < self.n:
            if it >= S:
                ok = ok and (yield self.empty[it % S], it // S - 1)
            if not ok and self.leaves:
                break
            self.put(it, 0)
            bar = self.listed[it % S]
            bar.tx += 1
            self.copying[it % S] = True
            bar.arrive()

            def land(bar=bar, it=it):
                self.copying[it % S] = False
                bar.tx -= 1
                bar.turn()
            self.queue(land)
            yield None
            it += 1
        if it == self.n:
            for k in range(it, it + 3):
                if k >= S:
                    ok = ok and (yield self.empty[k % S], k // S - 1)
            if ok or not self.leaves:
                for k in range(it, it + 3):
                    self.put(k, -1 - (k - it))
                self.listed[it % S].arrive()
                self.listed[(it + 1) % S].arrive()
                yield None
        for k in range(max(0, it - (5 if ok else 8)), it):
            ok = (yield self.listed[k % S], k // S) and ok

    def generator(self, g, w):
        S, it, ok = self.SLOTS, g, True
        while True:
            ok = ok and (yield self.listed[it % S], it // S)
            if it >= 3 and self.x_wait:
                ok = ok and (yield self.full[(it - 3) % self.nf], (it - 3) // self.nf)
            end = self.record(it) if ok else -4
            if end == 0:
                c, s, used, _ = self.steps[it]
                self.see(it < self.BUFS or self.done[it - self.BUFS], f"X of step {it - 3} overwritten early")
                if s == 0:
                    several = self.w_wait and used >= 0 and self.steps[used][1] > 0
                    if used >= 0 and it - used < 8 and (it - used > 3 or several):
                        ok = ok and (yield self.empty[used % S], used // S)
                    self.see(used < 0 or all(self.done[k] for k in range(used + 1) if self.steps[k][0] == c - self.BUFS),
                             f"W of chunk {c - self.BUFS} overwritten early")
                self.wrote[it] += 1
                yield None
            elif not ok and it < self.n:
                self.wrote[it] += 1          # past it, without a look at its record
            meet = self.meet[g]
            gen = meet.arrive(end < 0)
            yield lambda: meet.met(gen)
            if w == 0 and ok:
                self.ready[it % S].arrive()
                if end == -1:
                    self.ready[(it + 2) % S].arrive()
            if meet.stop[gen]:
                return
            it += 2

    def issuer(self, k):
        S, it, behind, ok = self.SLOTS, k, None, True
        while True:
            ok = yield self.ready[it % S], it // S
            if not ok or self.record(it) < 0:
                break
            c, s, _, _ = self.steps[it]
            if 1 <= s <= 3:
                ok = ok and (yield self.ready[(it - s) % S], (it - s) // S)
            if it >= self.DBUFS:
                ok = ok and (yield self.empty[(it - self.DBUFS) % S], (it - self.DBUFS) // S)
            if not ok:
                break
            self.see(it < self.DBUFS or self.read[it - self.DBUFS] == 8, f"sums of step {it - self.DBUFS} overwritten early")
            self.see(self.wrote[it] == 8 and self.wrote[it - s] == 8, f"MMAs of step {it} before its operands")
            self.issued[it] = True

            def land(it=it):
                self.done[it] = True
                self.full[it % self.nf].arrive()
            behind = self.queue(land, behind)
            yield None
            it += 3
        if it >= 3:
            yield self.full[(it - 3) % self.nf], (it - 3) // self.nf

    def adder(self, w):
        meets = 0
        for it in range(self.n):
            if not (yield self.full[it % self.nf], it // self.nf):
                return
            self.see(self.done[it], f"sums of step {it} read before they are complete")
            self.record(it)
            yield None
            self.read[it] += 1
            self.empty[it % self.SLOTS].arrive()
            if not self.steps[it][3]:
                continue
            # the end of a tile split between CTAs: planes summed, partial sums
            # stored, the tile's CTAs counted by thread 0, their sums read
            self.sums[w] = it
            for what in ("planes", "partial sums", "flag", "done")[: 4 if it + 1 < self.n else 3]:
                if what == "flag" and w == 0:
                    self.flag = it
                self.summed.arrive()
                ok = yield self.summed, meets
                meets += 1
                if not ok and self.adders_leave:
                    return
                if what == "planes":
                    check(all(x == it for x in self.sums), "another warp's sums read before they are written")
                if what == "flag":
                    check(self.flag == it, "the tile's CTAs read before thread 0 has counted them")
                yield None


class Forward(Model):
    """One CTA: steps of the given tiles (a number per step)."""

    def __init__(self, rng, tiles, leaves=FWD_LEAVES, fails=False):
        super().__init__(rng, fails)
        self.tiles, self.leaves = tiles, leaves
        n = self.n = len(tiles)
        self.full = [Barrier(1) for _ in range(2)]
        self.empty = [Barrier(8) for _ in range(4)]
        self.ready = [Barrier(1) for _ in range(4)]
        self.listed = [Barrier(1) for _ in range(4)]
        self.slot, self.copying = [None] * 4, [False] * 4
        self.wrote, self.read = [0] * n, [0] * n
        self.issued, self.done = [False] * n, [False] * n
        self.meets = [Meeting(8) for _ in range(2)]
        self.add("lister", self.lister())
        for k in range(2):
            self.add(f"issuer {k}", self.issuer(k))
        for w in range(8):
            self.add(f"generator {w}", self.generator(w))
            self.add(f"summer {w}", self.summer(w))

    def put(self, it, end):
        if 0 <= it - 4 < self.n:
            check(self.read[it - 4] == 8 and self.wrote[it - 4] == 8 and self.issued[it - 4], f"record of step {it - 4} rewritten early")
        check(not self.copying[it & 3], "a copy goes to a slot whose last copy is in flight")
        self.slot[it & 3] = (it, end)

    def record(self, it):
        check(self.slot[it & 3] is not None and self.slot[it & 3][0] == it, f"record of step {it} not there")
        return self.slot[it & 3][1]

    def lister(self):
        ok, it = True, 0
        while it < self.n:
            if it >= 4:
                ok = ok and (yield self.empty[it & 3], (it >> 2) - 1)
            if not ok and self.leaves:
                break
            self.put(it, False)
            bar = self.listed[it & 3]
            bar.tx += 1
            self.copying[it & 3] = True
            bar.arrive()

            def land(bar=bar, it=it):
                self.copying[it & 3] = False
                bar.tx -= 1
                bar.turn()
            self.queue(land)
            yield None
            it += 1
        if it == self.n:
            for k in (it, it + 1):
                if k >= 4:
                    ok = ok and (yield self.empty[k & 3], (k >> 2) - 1)
            if ok or not self.leaves:
                for k in (it, it + 1):
                    self.put(k, True)
                    self.listed[k & 3].arrive()
                yield None
        for k in range(max(0, it - (2 if ok else 4)), it):
            ok = (yield self.listed[k & 3], k >> 2) and ok

    def generator(self, w):
        it, ok = 0, True
        while True:
            ok = ok and (yield self.listed[it & 3], it >> 2)
            if it >= 2:
                ok = ok and (yield self.full[it & 1], (it >> 1) - 1)
            first, second = self.meets
            gen = first.arrive(not ok)
            yield lambda: first.met(gen)
            if first.stop[gen]:
                return
            if self.record(it):
                if w == 0:
                    self.ready[it & 3].arrive()
                return
            self.see(it < 2 or self.done[it - 2], f"A of step {it - 2} overwritten early")
            if it == 0 or self.tiles[it] != self.tiles[it - 1]:
                old = [k for k in range(it) if self.tiles[k] < self.tiles[it] - 1]
                self.see(all(self.done[k] for k in old), "B of an older tile overwritten early")
            self.wrote[it] += 1
            gen = second.arrive()
            yield lambda: second.met(gen)
            if w == 0:
                self.ready[it & 3].arrive()
            it += 1

    def issuer(self, d):
        it, behind, ok = d, None, True
        while True:
            ok = yield self.listed[it & 3], it >> 2
            if not ok or self.record(it):
                break
            ok = yield self.ready[it & 3], it >> 2
            if it >= 2:
                ok = ok and (yield self.empty[(it - 2) & 3], (it - 2) >> 2)
            if not ok:
                break
            self.see(it < 2 or self.read[it - 2] == 8, f"sums of step {it - 2} overwritten early")
            self.see(self.wrote[it] == 8, f"MMAs of step {it} before its operands")
            self.issued[it] = True

            def land(it=it):
                self.done[it] = True
                self.full[it & 1].arrive()
            behind = self.queue(land, behind)
            yield None
            it += 2
        if it >= 2:
            yield self.full[d], (it - 2) >> 1

    def summer(self, w):
        for it in range(self.n + 1):
            if not (yield self.ready[it & 3], it >> 2) or self.record(it):
                return
            if not (yield self.full[it & 1], it >> 1):
                return
            self.see(self.done[it], f"sums of step {it} read before they are complete")
            yield None
            self.read[it] += 1
            self.empty[it & 3].arrive()


def schedule(rng):
    chunks = [rng.choice([0, 0, 0, 1, 1, 2, 3, 5]) if rng.random() < 0.6 else 0 for _ in range(rng.randint(1, 14))]
    return chunks, {k for k in range(len(chunks)) if rng.random() < 0.4}


@pytest.mark.parametrize("seed", range(60))
def test_adjoint_roles(seed):
    rng = random.Random(seed)
    Adjoint(rng, *schedule(rng)).play()


def tiles_of(rng):
    tiles = [0]
    for _ in range(rng.randint(0, 24)):
        tiles.append(tiles[-1] + (rng.random() < 0.5))
    return tiles


@pytest.mark.parametrize("seed", range(40))
def test_forward_roles(seed):
    rng = random.Random(seed)
    Forward(rng, tiles_of(rng)).play()


@pytest.mark.parametrize("seed", range(60))
def test_every_role_ends_after_a_wait_that_ran_out(seed):
    rng = random.Random(seed)
    Adjoint(rng, *schedule(rng), fails=True).play()
    Forward(rng, tiles_of(rng), fails=True).play()


def caught(make):
    for seed in range(60):
        rng = random.Random(seed)
        try:
            make(rng).play()
        except Violation:
            return True
    return False


def test_planted_mistakes_are_caught():
    assert caught(lambda r: Adjoint(r, *schedule(r), nfull=4))
    assert caught(lambda r: Adjoint(r, *schedule(r), x_wait=False))
    assert caught(lambda r: Adjoint(r, *schedule(r), fails=True, leaves=False))
    assert caught(lambda r: Forward(r, tiles_of(r), fails=True, leaves=False))
    assert caught(lambda r: Adjoint(r, *schedule(r), fails=True, adders_leave=False))


# A chunk of two strips, then chunks of one: W's buffer is free again three
# steps after the second strip, whose MMAs another thread issued than the
# first strip's.
SHORT = [1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0]


@pytest.mark.parametrize("seed", range(40))
def test_first_strips_are_done_before_w_is_rewritten(seed):
    Adjoint(random.Random(seed), SHORT, set()).play()


def test_waiting_for_the_last_strip_alone_is_caught():
    assert caught(lambda r: Adjoint(r, SHORT, set(), w_wait=False))
