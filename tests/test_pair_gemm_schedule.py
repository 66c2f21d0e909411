"""The barrier protocol of the CTA-pair GEMM (tc_pair.cuh, gemm_pair) and its
tile walk, model-checked on the CPU.

Each CTA's TMA thread fills its own stages (after empty[s] of its CTA) and
counts the bytes on the leader's full[s], which also needs the leader's own
arrival (its expect_tx); the leader's MMA thread consumes a stage when both
CTAs' bytes are there and commits empty[s] and tfull to both CTAs; the eight
epilogue warps of each CTA arrive on the leader's tempty.  The model runs the
roles in random interleavings, with copies and commits completing after random
delays (a commit reaches the two CTAs at different times), and checks that
every role finishes, that no parity wait could see an aliased phase, that a
stage is refilled only after the MMAs that read it, and that the accumulators
are overwritten only after all sixteen warps read them."""
import random

import pytest


class Barrier:
    """Completes a phase when `count` arrivals and all expected bytes are in."""

    def __init__(self, count):
        self.count, self.pending, self.tx, self.done = count, count, 0, 0

    def _check(self):
        if self.pending == 0 and self.tx == 0:
            self.done += 1
            self.pending = self.count

    def arrive(self, expect=0):
        self.pending -= 1
        assert self.pending >= 0
        self.tx += expect
        self._check()

    def bytes(self, n):
        self.tx -= n
        self._check()


def ready(bar, phase):
    assert bar.done - phase <= 1, (bar.done, phase)      # an aliased parity wait
    return bar.done > phase


def run_pair(ntiles, nkb, stages, rng, mutant=None, warps=8):
    full = [Barrier(1) for _ in range(stages)]                       # leader's
    empty = [[Barrier(1) for _ in range(stages)] for _ in range(2)]
    tfull = [Barrier(1) for _ in range(2)]
    tempty = Barrier(2 * warps)                                      # leader's
    copies, commits, consumed = [], [], set()
    started, reads = set(), {}

    def producer(rank):
        it = 0
        for _ in range(ntiles):
            for _kb in range(nkb):
                s = it % stages
                if it >= stages and mutant != "no_empty_wait":
                    while not ready(empty[rank][s], it // stages - 1):
                        yield
                    assert it - stages in consumed
                if rank == 0:
                    full[s].arrive(expect=2)
                copies.append((rank, s, it))
                it += 1
                yield

    def mma():
        it = 0
        for tl in range(ntiles):
            if tl >= 1 and mutant != "no_tempty_wait":
                while not ready(tempty, tl - 1):
                    yield
                assert reads.get(tl - 1) == 2 * warps
            started.add(tl)
            for _kb in range(nkb):
                s = it % stages
                while not ready(full[s], it // stages):
                    yield
                commits.append(("empty", s, it))
                it += 1
                yield
            commits.append(("tfull", None, None))
            yield

    def epilogue(rank):
        for tl in range(ntiles):
            while not ready(tfull[rank], tl):
                yield
            assert tl + 1 not in started
            yield
            assert tl + 1 not in started
            reads[tl] = reads.get(tl, 0) + 1
            tempty.arrive()

    late = []                                             # the peer's half of a commit
    roles = [producer(0), producer(1), mma()] + [epilogue(k % 2) for k in range(2 * warps)]
    live = list(range(len(roles)))
    for _ in range(10 ** 6):
        if not live and not copies and not commits and not late:
            assert reads == {tl: 2 * warps for tl in range(ntiles)}
            return
        r = rng.random()
        if copies and r < 0.2:
            _, s, _ = copies.pop(rng.randrange(len(copies)))
            full[s].bytes(1)
            continue
        if late and r < 0.3:
            kind, s = late.pop(0)
            (empty[1][s] if kind == "empty" else tfull[1]).arrive()
            continue
        if commits and r < 0.4:
            kind, s, it = commits.pop(0)                  # in issue order
            if it is not None:
                consumed.add(it)
            (empty[0][s] if kind == "empty" else tfull[0]).arrive()
            late.append((kind, s))
            continue
        if live:
            k = rng.choice(live)
            try:
                next(roles[k])
            except StopIteration:
                live.remove(k)
    raise AssertionError("the roles did not finish (deadlock)")


@pytest.mark.parametrize("ntiles,nkb,stages", [(1, 1, 2), (1, 16, 2), (3, 1, 2), (4, 16, 2), (5, 2, 3),
                                               (4, 3, 3), (2, 7, 3)])
def test_pair_protocol(ntiles, nkb, stages):
    rng = random.Random(1000 * ntiles + 10 * nkb + stages)
    for _ in range(30):
        run_pair(ntiles, nkb, stages, rng)


@pytest.mark.parametrize("mutant", ["no_tempty_wait", "no_empty_wait"])
def test_model_catches_a_dropped_wait(mutant):
    rng = random.Random(5)
    with pytest.raises(AssertionError):
        for _ in range(200):
            run_pair(6, 4, 2, rng, mutant)


def items(nm, n64, pairs):
    """PairTiles: the work items (row tile, first 64-column group, groups)."""
    nn = (n64 + 1) // 2
    t = nm * nn
    rest = t % pairs
    full = t - rest if 2 * rest <= pairs else t
    out = []
    for k in range(full + 2 * (t - full)):
        tile = k if k < full else full + (k - full) // 2
        g0, ng = 2 * (tile % nn), 1 if n64 - 2 * (tile % nn) < 2 else 2
        if k >= full:
            g0, ng = (g0 + 1, ng - 1) if (k - full) & 1 else (g0, 1)
        out.append((tile // nn, g0, ng))
    return out


@pytest.mark.parametrize("pairs", [1, 5, 76])
@pytest.mark.parametrize("nm,n64", [(1, 1), (1, 16), (3, 5), (16, 4), (32, 16), (76, 1), (5, 31)])
def test_tiles_cover_the_output_once(nm, n64, pairs):
    """Also with the smaller grid a launch of fewer items uses (the walk is
    recomputed from the number of pairs launched)."""
    got = items(nm, n64, pairs)
    launched = min(pairs, len(got))
    for walk in (got, items(nm, n64, launched)):
        seen = [(tm, g0 + h) for tm, g0, ng in walk for h in range(ng)]
        assert sorted(seen) == [(tm, g) for tm in range(nm) for g in range(n64)]
