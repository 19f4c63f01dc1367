"""The tile rings of the two-step kernels (csrc/xrow.cuh, csrc/colpass.cuh) as a model on the CPU: their
warps, mbarriers and copies step by step in random order, with waits that run out at random.  Whatever the
order, no mbarrier is armed or arrived at beyond its count, no copy is under way when the block ends, every
warp ends, and a run in which no wait ran out has taken every tile; a wait that ran out is recorded.
`careless`: a copying warp that refills a set without looking whether a wait has given up, as k_col's did,
must be caught."""
from __future__ import annotations

import random

import pytest


class Fault(Exception):
    pass


class Bar:
    def __init__(self, count):
        self.count = self.pending = count
        self.tx = 0
        self.phase = 0

    def _turn(self):
        if self.pending == 0 and self.tx == 0:
            self.phase ^= 1
            self.pending = self.count

    def arrive(self, tx=0):
        if self.pending == 0:
            raise Fault("arrival beyond the count")
        self.tx += tx
        self.pending -= 1
        self._turn()

    def complete(self):
        self.tx -= 1
        self._turn()

    def passed(self, parity):   # test of the phase with this parity
        return self.phase != parity


class Block:
    def __init__(self, rng, p_out):
        self.rng, self.p_out = rng, p_out
        self.failed = self.err = False
        self.issued = 0
        self.flying = []          # mbarriers of copies under way
        self.ran_out = False
        self.taken = set()

    def out(self):                # does this poll use up the wait's limit?
        if self.rng.random() < self.p_out:
            self.ran_out = True
            return True
        return False

    def load(self, bar):
        bar.arrive(1)
        self.flying.append(bar)

    def give_up(self):
        self.failed = self.err = True

    def warp_wait(self, bar, parity):
        """Generator: True once over, False after giving up."""
        while not bar.passed(parity):
            if self.failed or self.out():
                self.give_up()
                return False
            yield
        return True

    def settle(self, full, sent, S):
        for i in range(max(0, sent - S), sent):
            while not full[i % S].passed((i // S) & 1):
                yield


def rows(b, n, S, T):
    """k_xrow: T teams of three warps, a producer."""
    full, empty, tbar = [Bar(1) for _ in range(S)], [Bar(3) for _ in range(S)], Bar(1)

    def producer():
        b.load(tbar)
        k, ph, sent = 0, 1, 0
        for _ in range(n):
            if not (yield from b.warp_wait(empty[k], ph)):
                break
            b.load(full[k])
            sent += 1
            b.issued = sent
            yield
            k += 1
            if k == S:
                k, ph = 0, ph ^ 1
        yield from b.settle(full, sent, S)
        while not tbar.passed(0):
            yield

    def warp(team, c):
        if not (yield from b.warp_wait(tbar, 0)):
            return
        for i in range(team, n, T):
            u, k = divmod(i, S)
            while b.issued <= i:
                if b.failed or b.out():
                    b.give_up()
                    return
                yield
            if not (yield from b.warp_wait(full[k], u & 1)):
                return
            b.taken.add((i, c))
            yield
            empty[k].arrive()

    return [producer()] + [warp(t, c) for t in range(T) for c in range(3)], 3 * n


def columns(b, n, S, NG, copy, careless):
    """k_col: NG groups of two warps, a copying warp (copy: it also stores the tiles)."""
    W = 2
    full, done, tbar = [Bar(1) for _ in range(S)], [Bar(W if copy else 1) for _ in range(S)], Bar(1)
    meet = [[0, 0] for _ in range(NG)]   # a group's barrier: arrivals, phase

    def tile_done(k, ph):
        ok = yield from b.warp_wait(done[k], ph)
        return ok and not b.failed

    def refill(k, ph):
        if careless:                     # goes on when a wait has given up
            while not (b.failed or done[k].passed(ph)):
                if b.out():
                    b.give_up()
                yield
            return True
        return (yield from tile_done(k, ph))

    def loader():
        b.load(tbar)

        def load(k):
            b.load(full[k])
            b.issued += 1
        for i in range(min(S, n)):
            load(i)
            yield
        k = kl = ph = 0
        ok = True
        if not copy:
            for _ in range(S, n):
                ok = yield from refill(k, ph)
                if not ok:
                    break
                load(k)
                yield
                k += 1
                if k == S:
                    k, ph = 0, ph ^ 1
        else:
            lag = 1 if S >= NG + 2 else 0
            for i in range(n):
                ok = yield from refill(k, ph)
                if not ok:
                    break
                yield                    # (the store, and the wait for its reads)
                if i >= lag and i - lag + S < n:
                    load(kl)
                    kl = (kl + 1) % S
                k += 1
                if k == S:
                    k, ph = 0, ph ^ 1
        if not ok or b.failed:
            yield from landed()

    def landed():
        yield from b.settle(full, b.issued, S)
        while not tbar.passed(0):
            yield

    def sync(g):
        m = meet[g]
        phase = m[1]
        m[0] += 1
        if m[0] == W:
            m[0], m[1] = 0, m[1] + 1
        while m[1] == phase:
            yield

    def wait(bar, parity):
        while not b.failed and not bar.passed(parity):
            if b.out():
                b.give_up()
            yield

    def warp(g, w):
        yield from wait(tbar, 0)
        for i in range(g, n, NG):
            u, k = divmod(i, S)
            while b.issued <= i and not b.failed:
                if b.out():
                    b.give_up()
                yield
            yield from wait(full[k], u & 1)
            if not b.failed:
                b.taken.add((i, w))
            yield
            yield from sync(g)
            if copy:
                done[k].arrive()
            else:
                yield from sync(g)
                if w == 0:
                    done[k].arrive()
        if not copy and b.failed:
            yield from landed()

    return [loader()] + [warp(g, w) for g in range(NG) for w in range(W)], W * n


def run(make, rng, p_out):
    b = Block(rng, p_out)
    alive, want = make(b)
    for _ in range(200000):
        if not alive:
            break
        if b.flying and rng.random() < 0.3:
            b.flying.pop(rng.randrange(len(b.flying))).complete()
            continue
        g = rng.choice(alive)
        try:
            next(g)
        except StopIteration:
            alive.remove(g)
    if alive:
        raise Fault("a warp does not end")
    if b.flying:
        raise Fault("a copy is under way at the end")
    assert b.err == b.ran_out
    if not b.ran_out:
        assert len(b.taken) == want


SHAPES = [(1, 3, 2), (2, 3, 2), (7, 3, 2), (11, 4, 2), (20, 8, 5), (13, 5, 4), (9, 3, 1)]


@pytest.mark.parametrize("n,S,T", SHAPES)
@pytest.mark.parametrize("p_out", [0.0, 0.002, 0.03, 0.3])
def test_row_kernel(n, S, T, p_out):
    for seed in range(60):
        run(lambda b: rows(b, n, S, min(T, S - 1)), random.Random(seed), p_out)


@pytest.mark.parametrize("n,S,NG", SHAPES)
@pytest.mark.parametrize("copy", [False, True])
@pytest.mark.parametrize("p_out", [0.0, 0.002, 0.03, 0.3])
def test_column_kernels(n, S, NG, copy, p_out):
    for seed in range(60):
        run(lambda b: columns(b, n, S, NG, copy, False), random.Random(seed), p_out)


@pytest.mark.parametrize("copy", [False, True])
def test_a_careless_copying_warp_is_caught(copy):
    with pytest.raises(Fault):
        for seed in range(200):
            run(lambda b: columns(b, 20, 4, 3, copy, True), random.Random(seed), 0.03)
