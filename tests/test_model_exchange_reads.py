"""CPU model of the exchange of the tridiagonal reduction (values that are their
own flags, eight buffers in turn, unset four steps ahead) with loads that may be
served early as well as stores that may be seen late.

A block at step t: wait for everyone's partial of step t-1, take everyone's words of
that step; a fence of the warp that publishes the partials, behind which nothing
stored before stays unseen; publish the step's word and partial, unset the word of
step t+4's buffer; a fence of the warps that read the partials, behind which (and the
step's last barrier) no load of the next step is served early."""
import random

import pytest

BUFS, AHEAD = 8, 4


def run(blocks, steps, seed, acquire):
    """True when every word taken is the one looked for."""
    rng = random.Random(seed)
    hist = {}                     # (kind, slot, block) -> [(time, value)], what memory held
    for k in ("word", "part"):
        for s in range(BUFS):
            for b in range(blocks):
                hist[k, s, b] = [(0, None)]
    pending = [[] for _ in range(blocks)]     # stores not yet seen, any order between fences
    since = [0] * blocks                       # time of the block's last reading fence
    pc = [("part", 0, 0)] * blocks
    end, now = 0, 0

    def load(g, key):
        now_v = hist[key][-1][1]
        if rng.random() < 0.5:
            return now_v
        at = rng.randint(since[g], now)        # served early
        return [v for tm, v in hist[key] if tm <= at][-1]

    while end < blocks:
        now += 1
        assert now < 3_000_000
        g = rng.randrange(blocks)
        if pending[g] and rng.random() < 0.25:
            key, v = pending[g].pop(rng.randrange(len(pending[g])))
            hist[key].append((now, v))
            continue
        what, t, i = pc[g]
        if what == "end":
            continue
        if what in ("part", "word"):
            if t == 0 or i == blocks:
                pc[g] = ("word", t, 0) if what == "part" else ("fence", t, 0)
                continue
            v = load(g, (what, (t - 1) % BUFS, i))
            if v is None:
                continue
            if v != (t - 1, i):
                return False
            pc[g] = (what, t, i + 1)
        elif what == "fence":
            if pending[g]:
                continue                       # what was stored before is seen first
            pc[g] = ("store", t, 0)
        elif what == "store":
            if t + AHEAD < steps:
                pending[g] += [((k, (t + AHEAD) % BUFS, g), None) for k in ("word", "part")]
            pending[g] += [((k, t % BUFS, g), (t, g)) for k in ("word", "part")]
            pc[g] = ("acquire", t, 0)
        else:
            if acquire:
                since[g] = now                 # later loads stay behind
            if t + 1 == steps:
                pc[g] = ("end", t, 0)
                end += 1
            else:
                pc[g] = ("part", t + 1, 0)
    return True


@pytest.mark.parametrize("blocks,steps", [(2, 40), (3, 40), (5, 30)])
def test_the_fences_of_a_step_order_the_exchange(blocks, steps):
    assert all(run(blocks, steps, seed, True) for seed in range(60))


def test_ordered_stores_alone_are_not_enough():
    """A fence that orders the stores only: a word of eight steps ago passes for a
    new one."""
    assert not all(run(3, 40, seed, False) for seed in range(60))
