"""What the epilogue warps of the CTA-pair GEMM (tc_pair.cuh, gemm_pair) do
when a wait runs out, model-checked on the CPU.

The two warps of a lane quarter meet in a named barrier without a time limit
to exchange sums, so neither may reach it when the other has left.  Each times
its own wait for a tile: near the limit one may run out while the other's
succeeds.  The model gives every wait a random outcome and checks that both
warps always finish, whatever the interleaving and the kinds of the items
(128 columns: no exchange; 64 columns: two barriers).  The second model looks at how long a
correct run waits."""
import random

import pytest


class Named:
    """A named barrier of two warps; join() returns a function that tells
    whether the barrier has completed, and the AND of the values brought."""

    def __init__(self):
        self.round, self.arrived, self.value, self.results = 0, 0, True, []

    def join(self, value=True):
        me = self.round
        self.arrived += 1
        self.value = self.value and value
        if self.arrived == 2:
            self.results.append(self.value)
            self.round, self.arrived, self.value = me + 1, 0, True
        return lambda: (self.round > me, self.results[me] if self.round > me else None)


def run_quarter(items, rng, agree=True):
    bar = Named()
    done, wanted, failed = [], {}, []

    def meet(value=True):
        poll = bar.join(value)
        while not poll()[0]:
            yield None
        yield poll()[1]

    def warp(w):
        for k, ng in enumerate(items):
            ok = rng.random() > 0.15                 # the wait for the tile
            yield
            if agree:
                for ok in meet(ok):
                    if ok is None:
                        yield
            if not ok:
                failed.append(w)
                break
            if ng == 1:
                for _ in range(2):                   # write, meet, read, meet
                    for r in meet():
                        if r is None:
                            yield
            done.append((w, k))
        wanted[w] = True

    roles = {w: warp(w) for w in range(2)}
    for _ in range(10000):
        if not roles:
            return done, failed
        w = rng.choice(list(roles))
        try:
            next(roles[w])
        except StopIteration:
            del roles[w]
    raise AssertionError("a warp waits for one that has left")


@pytest.mark.parametrize("items", [[1], [2, 1], [2, 2, 1, 1], [1] * 6, [2] * 5])
def test_both_warps_leave_together(items):
    rng = random.Random(len(items))
    for _ in range(500):
        done, failed = run_quarter(items, rng)
        assert sorted(k for w, k in done if w == 0) == sorted(k for w, k in done if w == 1)
        assert len(failed) in (0, 2)


def test_the_model_sees_a_warp_that_leaves_alone():
    rng = random.Random(3)
    with pytest.raises(AssertionError):
        for _ in range(500):
            run_quarter([2, 1, 1], rng, agree=False)


def longest_wait(ntiles, tile_time, after_roles):
    """Longest wait of the peer CTA in a run whose tiles complete every
    `tile_time`: its epilogue waits tile by tile, its warp 1 for the leader's
    last commit, from the end of the CTA's roles or from the kernel's start."""
    finished = [(t + 1) * tile_time for t in range(ntiles)]
    waits, now = [], 0.0
    for t in finished:
        waits.append(t - now)
        now = max(now, t)
    last_commit = finished[-1]
    waits.append(max(0.0, last_commit - (now if after_roles else 0.0)))
    return max(waits)


@pytest.mark.parametrize("ntiles", [1, 7, 1000])
def test_no_wait_spans_more_than_one_tile(ntiles):
    """The limit of a wait is one for a step, however many tiles a call has."""
    assert longest_wait(ntiles, 0.25, after_roles=True) <= 0.25
    assert longest_wait(1000, 0.25, after_roles=False) > 2.0
