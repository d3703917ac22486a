"""Blocks of a pair leave a launch in which a wait was abandoned: no copy may be under way between them any more (no GPU needed; a run that
gives up is not made on one).  The two blocks are acted out step by step, with copies that take any time and waits given up anywhere; what
they wait for before they leave is the library's own decision (sdv_debug_pair_debt)."""
import numpy as np
import pytest

from paper_2510_15312_b200.binding import EINVAL, pair_debt

LAYERS, WARPS = 5, 8


class Barrier:
    """An mbarrier of WARPS arrivals; bytes may be counted before they are expected."""

    def __init__(self):
        self.done, self.pending, self.tx = 0, WARPS, 0

    def update(self, arrivals, tx):
        assert arrivals <= self.pending, "more arrivals than the phase takes"
        self.pending -= arrivals
        self.tx += tx
        if self.pending == 0 and self.tx == 0:
            self.done, self.pending = self.done + 1, WARPS

    def over(self, phase):
        """A wait by parity: tells the running phase from the one before it, no more."""
        assert phase in (self.done - 1, self.done)
        return self.done > phase


class Block:
    def __init__(self):
        self.bar, self.mine, self.abort, self.arrived, self.left = Barrier(), 0, False, 0, False


def act_out(rng, drains):
    """Copies still under way when a block left."""
    a, b = Block(), Block()
    flying = []                                    # [receiver, steps to go]
    give_up = rng.choice([0.0, 0.02, 0.2])
    lost = 0

    def life(me, other):
        def waits(done):                           # a bounded wait
            while not done():
                if me.abort or rng.random() < 0.01 + give_up:
                    me.abort = True
                    return False
                yield
            return True
        for layer in range(LAYERS):
            me.arrived += 1                        # the grid barrier in front: met whatever happened
            yield from waits(lambda: other.arrived > layer)
            if me.abort:
                continue                           # the phase does no work
            if rng.random() < give_up / 4:
                me.abort = True                    # some other wait of the phase: the columns are sent all the same
            me.bar.update(WARPS, 1)                # one arrival expects the other's bytes
            flying.append([other, int(rng.integers(0, 12))])
            me.mine += 1
            yield
            if not me.abort:
                yield from waits(lambda: me.bar.over(layer))
        me.arrived = LAYERS + 1
        while other.arrived <= LAYERS:             # first cluster barrier
            yield
        assert abs(me.mine - other.mine) <= 1
        if me.abort or other.abort:
            debt = pair_debt(me.mine, other.mine) if drains else 0
            if debt & 1:
                while not me.bar.over(me.mine - 1):
                    yield
            if debt & 2:
                me.bar.update(WARPS, 1)
                while not me.bar.over(me.mine):
                    yield
            me.arrived = LAYERS + 2
            while other.arrived <= LAYERS + 1:     # until the other one is done waiting too
                yield
        me.left = True

    running = [life(a, b), life(b, a)]
    if rng.random() < 0.5:
        running.reverse()
    for _ in range(5000):
        for g in list(running):
            if rng.random() < 0.7:
                try:
                    next(g)
                except StopIteration:
                    running.remove(g)
        lost += sum(a.left or b.left for _ in flying)
        for c in list(flying):
            c[1] -= 1
            if c[1] < 0:
                flying.remove(c)
                c[0].bar.update(0, -1) if not c[0].left else None
        if not running and not flying:
            return lost, a.abort or b.abort, abs(a.mine - b.mine)
    raise AssertionError("a block never left")


def test_no_copy_is_under_way_when_a_block_leaves():
    rng = np.random.default_rng(7)
    aborted, uneven, lost_without = 0, 0, 0
    for _ in range(3000):
        lost, gave_up, apart = act_out(rng, True)
        assert lost == 0
        aborted += gave_up
        uneven += apart
    for _ in range(500):
        lost_without += act_out(rng, False)[0] > 0
    assert aborted > 1000 and uneven > 100 and lost_without > 10   # such runs occur, and without the waits they leave copies behind


@pytest.mark.parametrize("mine,sent,want", [(0, 0, 0), (0, 1, 2), (1, 0, 0), (1, 1, 1), (1, 2, 3), (28, 27, 0), (28, 28, 1), (28, 29, 3), (-1, 0, EINVAL)])
def test_what_is_waited_for(mine, sent, want):
    assert pair_debt(mine, sent) == want
