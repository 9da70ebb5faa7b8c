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

The numbers of barriers are read from the sources. Mistakes planted in the
model (four barriers for the adjoint's MMAs, which the generators' wait can
find two phases on; an operand buffer taken back early) have to be caught.
"""
import pathlib
import random
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2505_08777_gb300" / "csrc"


def constant(name, file):
    return int(re.search(rf"\b{name} = (\d+)", (CSRC / file).read_text()).group(1))


ADJ_FULL = constant("kAdjFull", "sep_adjoint.cu")


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
    """A named barrier of n warps (bar.sync, barrier.red)."""

    def __init__(self, n):
        self.n, self.come, self.gen = n, 0, 0

    def arrive(self):
        self.come += 1
        if self.come == self.n:
            self.come, self.gen = 0, self.gen + 1
            return self.gen
        return self.gen + 1


class Model:
    def __init__(self, rng):
        self.rng, self.procs, self.later = rng, {}, []

    def add(self, name, gen):
        self.procs[name] = [gen, None]

    def queue(self, what, after=None):
        """An asynchronous completion, in order behind `after`."""
        item = [what, after]
        self.later.append(item)
        return item

    def play(self):
        speed = {n: 10 ** self.rng.uniform(-2, 0) for n in self.procs}
        speed["async"] = 10 ** self.rng.uniform(-2, 0)
        for gen in self.procs.values():
            gen[1] = next(gen[0], "end")
        while True:
            live = [n for n, g in self.procs.items() if g[1] != "end"]
            ready = [n for n in live if self.procs[n][1] is None or self.procs[n][1]()]
            land = [x for x in self.later if x[1] is None or x[1] not in self.later]
            if not live:
                return
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
                g = self.procs[pick]
                g[1] = next(g[0], "end")


def wait(bar, phase):
    return lambda: bar.passed(phase)


class Adjoint(Model):
    """One CTA: chunks of 2^ls strips, tiles ending after the chunks in `ends`."""

    SLOTS, BUFS, DBUFS = 8, 3, 4

    def __init__(self, rng, chunks, ends, nfull=ADJ_FULL, x_wait=True, w_wait=True):
        super().__init__(rng)
        self.nf, self.x_wait, self.w_wait = nfull, x_wait, w_wait
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
        self.wrote = [0] * n                 # generator warps done with a step's operands
        self.issued, self.done = [False] * n, [False] * n
        self.read = [0] * n                  # adder warps done with a step's sums
        self.left = {}                       # steps past which a role is
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
        self.slot[it % self.SLOTS] = (it, end)

    def record(self, it):
        check(self.slot[it % self.SLOTS] is not None and self.slot[it % self.SLOTS][0] == it, f"record of step {it} not there")
        return self.slot[it % self.SLOTS][1]

    def lister(self):
        S = self.SLOTS
        for it in range(self.n):
            if it >= S:
                yield wait(self.empty[it % S], it // S - 1)
            self.put(it, 0)
            bar = self.listed[it % S]
            bar.tx += 1
            bar.arrive()

            def land(bar=bar):
                bar.tx -= 1
                bar.turn()
            self.queue(land)
            yield None
        it = self.n
        for k in range(it, it + 3):
            if k >= S:
                yield wait(self.empty[k % S], k // S - 1)
        for k in range(it, it + 3):
            self.put(k, -1 - (k - it))
        self.listed[it % S].arrive()
        self.listed[(it + 1) % S].arrive()
        yield None
        for k in range(max(0, it - 5), it):
            yield wait(self.listed[k % S], k // S)

    def generator(self, g, w):
        S, it = self.SLOTS, g
        while True:
            yield wait(self.listed[it % S], it // S)
            if it >= 3 and self.x_wait:
                yield wait(self.full[(it - 3) % self.nf], (it - 3) // self.nf)
            end = self.record(it)
            if end == 0:
                c, s, used, _ = self.steps[it]
                check(it < self.BUFS or self.done[it - self.BUFS], f"X of step {it - 3} overwritten early")
                if s == 0:
                    several = self.w_wait and used >= 0 and self.steps[used][1] > 0
                    if used >= 0 and it - used < 8 and (it - used > 3 or several):
                        yield wait(self.empty[used % S], used // S)
                    check(used < 0 or all(self.done[k] for k in range(used + 1) if self.steps[k][0] == c - self.BUFS),
                          f"W of chunk {c - self.BUFS} overwritten early")
                self.wrote[it] += 1
                yield None
            gen = self.meet[g].arrive()
            yield lambda: self.meet[g].gen >= gen
            if w == 0:
                self.ready[it % S].arrive()
                if end == -1:
                    self.ready[(it + 2) % S].arrive()
            if end < 0:
                return
            it += 2

    def issuer(self, k):
        S, it, behind = self.SLOTS, k, None
        while True:
            yield wait(self.ready[it % S], it // S)
            if self.record(it) < 0:
                break
            c, s, _, _ = self.steps[it]
            if 1 <= s <= 3:
                yield wait(self.ready[(it - s) % S], (it - s) // S)
            if it >= self.DBUFS:
                yield wait(self.empty[(it - self.DBUFS) % S], (it - self.DBUFS) // S)
                check(self.read[it - self.DBUFS] == 8, f"sums of step {it - self.DBUFS} overwritten early")
            check(self.wrote[it] == 8 and self.wrote[it - s] == 8, f"MMAs of step {it} before its operands")
            self.issued[it] = True

            def land(it=it):
                self.done[it] = True
                self.full[it % self.nf].arrive()
            behind = self.queue(land, behind)
            yield None
            it += 3
        if it >= 3:
            yield wait(self.full[(it - 3) % self.nf], (it - 3) // self.nf)

    def adder(self, w):
        meets = 0
        for it in range(self.n):
            yield wait(self.full[it % self.nf], it // self.nf)
            check(self.done[it], f"sums of step {it} read before they are complete")
            self.record(it)
            yield None
            self.read[it] += 1
            self.empty[it % self.SLOTS].arrive()
            if self.steps[it][3]:
                for _ in range(2 if it + 1 < self.n else 1):
                    self.summed.arrive()
                    yield wait(self.summed, meets)
                    meets += 1


class Forward(Model):
    """One CTA: steps of the given tiles (a number per step)."""

    def __init__(self, rng, tiles):
        super().__init__(rng)
        self.tiles = tiles
        n = self.n = len(tiles)
        self.full = [Barrier(1) for _ in range(2)]
        self.empty = [Barrier(8) for _ in range(4)]
        self.ready = [Barrier(1) for _ in range(4)]
        self.listed = [Barrier(1) for _ in range(4)]
        self.slot = [None] * 4
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
        self.slot[it & 3] = (it, end)

    def record(self, it):
        check(self.slot[it & 3] is not None and self.slot[it & 3][0] == it, f"record of step {it} not there")
        return self.slot[it & 3][1]

    def lister(self):
        for it in range(self.n):
            if it >= 4:
                yield wait(self.empty[it & 3], (it >> 2) - 1)
            self.put(it, False)
            bar = self.listed[it & 3]
            bar.tx += 1
            bar.arrive()

            def land(bar=bar):
                bar.tx -= 1
                bar.turn()
            self.queue(land)
            yield None
        for k in (self.n, self.n + 1):
            if k >= 4:
                yield wait(self.empty[k & 3], (k >> 2) - 1)
            self.put(k, True)
            self.listed[k & 3].arrive()
        yield None
        for k in range(max(0, self.n - 2), self.n):
            yield wait(self.listed[k & 3], k >> 2)

    def generator(self, w):
        it = 0
        while True:
            yield wait(self.listed[it & 3], it >> 2)
            if it >= 2:
                yield wait(self.full[it & 1], (it >> 1) - 1)
            gen = self.meets[0].arrive()
            yield lambda: self.meets[0].gen >= gen
            if self.record(it):
                if w == 0:
                    self.ready[it & 3].arrive()
                return
            check(it < 2 or self.done[it - 2], f"A of step {it - 2} overwritten early")
            if it == 0 or self.tiles[it] != self.tiles[it - 1]:
                old = [k for k in range(it) if self.tiles[k] < self.tiles[it] - 1]
                check(all(self.done[k] for k in old), "B of an older tile overwritten early")
            self.wrote[it] += 1
            gen = self.meets[1].arrive()
            yield lambda: self.meets[1].gen >= gen
            if w == 0:
                self.ready[it & 3].arrive()
            it += 1

    def issuer(self, d):
        it, behind = d, None
        while True:
            yield wait(self.listed[it & 3], it >> 2)
            if self.record(it):
                break
            yield wait(self.ready[it & 3], it >> 2)
            if it >= 2:
                yield wait(self.empty[(it - 2) & 3], (it - 2) >> 2)
                check(self.read[it - 2] == 8, f"sums of step {it - 2} overwritten early")
            check(self.wrote[it] == 8, f"MMAs of step {it} before its operands")
            self.issued[it] = True

            def land(it=it):
                self.done[it] = True
                self.full[it & 1].arrive()
            behind = self.queue(land, behind)
            yield None
            it += 2
        if it >= 2:
            yield wait(self.full[d], (it - 2) >> 1)

    def summer(self, w):
        for it in range(self.n + 1):
            yield wait(self.ready[it & 3], it >> 2)
            if self.record(it):
                return
            yield wait(self.full[it & 1], it >> 1)
            check(self.done[it], f"sums of step {it} read before they are complete")
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


@pytest.mark.parametrize("seed", range(40))
def test_forward_roles(seed):
    rng = random.Random(seed)
    tiles = [0]
    for _ in range(rng.randint(0, 24)):
        tiles.append(tiles[-1] + (rng.random() < 0.5))
    Forward(rng, tiles).play()


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


# A chunk of two strips, then chunks of one: W's buffer is free again three
# steps after the second strip, whose MMAs another thread issued than the
# first strip's.
SHORT = [1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0]


@pytest.mark.parametrize("seed", range(40))
def test_first_strips_are_done_before_w_is_rewritten(seed):
    Adjoint(random.Random(seed), SHORT, set()).play()


def test_waiting_for_the_last_strip_alone_is_caught():
    assert caught(lambda r: Adjoint(r, SHORT, set(), w_wait=False))
