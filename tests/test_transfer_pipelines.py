"""CPU model of the synchronisation of the two tensor-core Lagrange transfers, k_lag_pairs and k_lag_targets: index
warps, copying warps, the MMA thread, the accumulator warps and the asynchronous completions of their copies and
MMAs, over random interleavings.

mbarriers follow the hardware's parity rule: a wait for phase k succeeds iff the number of completed phases has a
parity other than k's, so a barrier two phases ahead of a wait looks incomplete.  The model checks that no schedule
deadlocks, that no wait sees its barrier two phases ahead, that every MMA reads the chunk and every reader the row
numbers and accumulator fill that it expects, and that after a give-up at any wait every started copy has landed and
every issued MMA is done when the block ends."""
import random

import pytest


class Bar:
    def __init__(self, count):
        self.count, self.here, self.phase = count, 0, 0

    def arrive(self):
        self.here += 1
        assert self.here <= self.count, "more arrivals than the barrier's count"
        if self.here == self.count:
            self.here, self.phase = 0, self.phase + 1

    def test(self, k):
        ok = (self.phase & 1) != (k & 1)
        assert not ok or self.phase == k + 1, "phase %d seen while waiting for %d" % (self.phase, k)
        return ok


class Block:
    """One thread block: `units` units of `chunks` stage fills each, an accumulator fill every `part` stages.  With
    drain > 0 (k_lag_targets) a unit is one stage and an accumulator fill spans `drain` units."""

    def __init__(self, seed, units, chunks, part, nstg, ring, epw, drain=0, give_up=None, ix_arrivals=None):
        self.rnd, self.units, self.chunks, self.part = random.Random(seed), units, chunks, part
        self.nstg, self.ring, self.epw, self.drain, self.give_up = nstg, ring, epw, drain, give_up
        self.full = [Bar(5) for _ in range(nstg)]  # four copying warps, the operator copy's expect
        self.empty = [Bar(1) for _ in range(nstg)]
        self.accfull, self.accempty = [Bar(1), Bar(1)], [Bar(epw), Bar(epw)]
        readers = 4 if drain else 4 + epw
        self.ixfull = [Bar(1) for _ in range(ring)]
        self.ixempty = [Bar(readers if ix_arrivals is None else ix_arrivals) for _ in range(ring)]
        self.ix = [None] * ring            # unit whose row numbers a slot holds
        self.stage = [[None] * 5 for _ in range(nstg)]  # what each warp's copy, and the operator copy, left
        self.acc = [None, None]            # fill held by an accumulator
        self.copies = []                   # (unordered) copies in flight: callables
        self.tensor = []                   # MMAs and commits, in order
        self.bad = False                   # someone gave up: every other wait may run out too
        self.waits, self.cmax, self.at_barrier, self.any_bad = 0, 0, 0, False

    def wait(self, bar, k):
        """Generator; True, or False after a give-up."""
        self.waits += 1
        mine = self.waits
        while True:
            if self.give_up == mine:
                self.bad = True
                return False
            if bar.test(k):
                return True
            if self.bad and self.rnd.random() < 0.2:
                return False
            yield

    def fills(self):
        """(unit, first stage, end) of each accumulator fill, as the MMA thread makes them."""
        if self.drain:
            return [list(range(a, min(a + self.drain, self.units))) for a in range(0, self.units, self.drain)]
        return [list(range(u * self.chunks + k, u * self.chunks + min(k + self.part, self.chunks)))
                for u in range(self.units) for k in range(0, self.chunks, self.part)]

    def index(self, w):
        for u in range(w, self.units, 4):
            s = u % self.ring
            if u >= self.ring and not (yield from self.wait(self.ixempty[s], u // self.ring - 1)):
                return
            self.ix[s] = u
            yield
            self.ixfull[s].arrive()

    def copy(self, w):
        c, ok = 0, True

        def land(slot, part, tag, bar):
            self.stage[slot][part] = tag
            bar.arrive()

        for u in range(self.units):
            s = u % self.ring
            if not (yield from self.wait(self.ixfull[s], u // self.ring)):
                ok = False
                break
            assert self.ix[s] == u
            yield
            self.ixempty[s].arrive()
            for _ in range(self.chunks):
                slot = c % self.nstg
                if c >= self.nstg and not (yield from self.wait(self.empty[slot], c // self.nstg - 1)):
                    ok = False
                    break
                self.copies.append(lambda slot=slot, c=c: land(slot, w, c, self.full[slot]))
                if w == 0:
                    self.copies.append(lambda slot=slot, c=c: land(slot, 4, c, self.full[slot]))
                c += 1
                yield
            if not ok:
                break
        # after a give-up: all arrive on every stage any of them started
        self.any_bad |= not ok
        self.cmax = max(self.cmax, c)
        self.at_barrier += 1
        while self.at_barrier < 4:
            yield
        if self.any_bad:
            for d in range(c, self.cmax):
                self.full[d % self.nstg].arrive()
                if w == 0:
                    self.full[d % self.nstg].arrive()
            c = self.cmax
        if w == 0:
            for d in range(max(0, c - self.nstg), c):
                while not self.full[d % self.nstg].test(d // self.nstg):
                    yield

    def mma(self):
        ok = True
        for f, stages in enumerate(self.fills()):
            buf = f & 1
            if f >= 2 and not (yield from self.wait(self.accempty[buf], (f >> 1) - 1)):
                break
            for c in stages:
                slot = c % self.nstg
                if not (yield from self.wait(self.full[slot], c // self.nstg)):
                    ok = False
                    break

                def run(slot=slot, c=c, f=f, buf=buf):
                    # (after a give-up the products mean nothing: the error flag is up)
                    assert self.bad or self.stage[slot] == [c] * 5, "MMA of chunk %d reads %r" % (c, self.stage[slot])
                    self.acc[buf] = f

                self.tensor += [run, self.empty[slot].arrive]
                yield
            if not ok:
                break
            self.tensor.append(self.accfull[buf].arrive)
        done = []
        self.tensor.append(lambda: done.append(1))
        while not done:
            yield

    def epilogue(self, w):
        f = 0
        per_unit = 1 if self.drain else -(-self.chunks // self.part)
        for u in range(len(self.fills()) if self.drain else self.units):
            if not self.drain:
                s = u % self.ring
                if not (yield from self.wait(self.ixfull[s], u // self.ring)):
                    return
                assert self.ix[s] == u
                yield
                self.ixempty[s].arrive()
            for _ in range(per_unit):
                if not (yield from self.wait(self.accfull[f & 1], f >> 1)):
                    return
                assert self.bad or self.acc[f & 1] == f
                yield
                assert self.bad or self.acc[f & 1] == f, "accumulator refilled while it was read"
                self.accempty[f & 1].arrive()
                f += 1

    def run(self):
        live = [self.index(w) for w in range(4)] + [self.copy(w) for w in range(4)] + [self.mma()]
        live += [self.epilogue(w) for w in range(self.epw)]
        idle = 0
        while live:
            idle += 1
            assert idle < 200000, "no progress: deadlock"
            r = self.rnd.random()
            if self.copies and r < 0.25:
                self.copies.pop(self.rnd.randrange(len(self.copies)))()
                idle = 0
            elif self.tensor and r < 0.5:
                self.tensor.pop(0)()
                idle = 0
            else:
                g = self.rnd.choice(live)
                before = (self.waits, len(self.copies), len(self.tensor))
                try:
                    next(g)
                except StopIteration:
                    live.remove(g)
                    idle = 0
                if before != (self.waits, len(self.copies), len(self.tensor)):
                    idle = 0
        assert not self.copies and not self.tensor, "copies or MMAs outlive the block"
        return self.waits


# stages, K chunks per unit (in stages), stages per accumulator fill, accumulator warps
PAIRS = [(4, 1, 1, 4), (4, 4, 4, 4), (8, 1, 1, 4), (6, 4, 4, 4), (4, 7, 7, 4), (4, 48, 48, 4), (5, 14, 4, 8),
         (5, 1, 4, 8), (5, 4, 4, 8), (5, 32, 4, 8), (5, 5, 4, 8)]
TARGETS = [(4, 8), (8, 8)]


@pytest.mark.parametrize("units", [0, 1, 2, 3, 4, 5, 9, 23])
@pytest.mark.parametrize("nstg,chunks,part,epw", PAIRS)
def test_transfer_by_translation(nstg, chunks, part, epw, units):
    if units * chunks > 400:
        pytest.skip("covered by the shorter units")
    for seed in range(4):
        Block(seed, units, chunks, part, nstg, 4, epw).run()


@pytest.mark.parametrize("steps", [1, 2, 7, 8, 9, 15, 16, 17, 24, 33, 100])
@pytest.mark.parametrize("nstg,drain", TARGETS)
def test_target_stationary_transfer(nstg, drain, steps):
    for seed in range(4):
        Block(seed, steps, 1, 1, nstg, 8, 4, drain=drain).run()


@pytest.mark.parametrize("kw", [dict(units=6, chunks=3, part=2, nstg=5, ring=4, epw=8),
                                dict(units=7, chunks=1, part=1, nstg=4, ring=4, epw=4),
                                dict(units=20, chunks=1, part=1, nstg=4, ring=8, epw=4, drain=8)])
def test_give_up_at_every_wait(kw):
    n = Block(0, **kw).run()
    for k in range(1, n + 1):
        for seed in range(3):
            Block(seed, give_up=k, **kw).run()


def test_model_catches_a_wrong_arrival_count():
    with pytest.raises(AssertionError):
        for seed in range(20):
            Block(seed, 12, 2, 2, 4, 4, 4, ix_arrivals=7).run()


def test_model_catches_a_missing_compensation():
    class NoCompensation(Block):
        def copy(self, w):
            for x in Block.copy(self, w):
                if self.at_barrier == 4:
                    self.any_bad = False
                yield x

    with pytest.raises(AssertionError):
        for k in range(1, 60):
            for seed in range(4):
                NoCompensation(seed, 6, 3, 2, 5, 4, 8, give_up=k).run()
