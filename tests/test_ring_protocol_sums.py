"""The ring model of test_ring_protocol.py with the warp that adds up z (64 tokens): it waits for
fullB[s] in every round and then arrives on empty[s], which takes that arrival and the issuer's
commit.  At every wait the barrier is at the awaited phase or one past it, every round's MMAs run
once, and a stage's activation tile is not loaded again before the warp has read it."""
import random

import pytest

from test_ring_protocol import Bar, wait


def run(seed, S, NI):
    rnd = random.Random(seed)
    rounds = [p for p in (0, 1, 2) for _ in range(rnd.randint(0, 4)) for _ in range(rnd.randint(0, 12))]
    full_a = [Bar(1, f"fullA{s}") for s in range(S)]
    full_b = [Bar(1, f"fullB{s}") for s in range(S)]
    empty = [Bar(2, f"empty{s}") for s in range(S)]
    cfull = [Bar(1, f"cfull{s}") for s in range(S)]
    landing, mma, loaded, read = [], [], [-1] * S, []

    def delay():
        for _ in range(rnd.randint(0, 4)):
            yield

    def producer(weights):
        for r, p in enumerate(rounds):
            s = r % S
            if r >= S:
                yield from wait(empty[s], r // S - 1, "producer")
            yield from delay()
            if not weights:
                loaded[s] = r
                landing.append([rnd.randint(1, 20), full_b[s]])
            elif p == 1:
                cfull[s].arrive()
            else:
                landing.append([rnd.randint(1, 20), full_a[s]])

    def decoder(d):
        seen = [0] * S
        for r, p in enumerate(rounds):
            s = r % S
            if s % 4 == d and p == 1:
                yield from wait(cfull[s], seen[s], f"decoder {d}")
                seen[s] += 1
                yield from delay()
                full_a[s].arrive()

    def issuer(q):
        for r, _ in enumerate(rounds):
            s = r % S
            if s % NI == q:
                yield from wait(full_a[s], r // S, f"issuer {q}")
                yield from wait(full_b[s], r // S, f"issuer {q}")
                mma.append(r)
                landing.append([rnd.randint(1, 10), empty[s]])

    def sums():
        for r, _ in enumerate(rounds):
            s = r % S
            yield from wait(full_b[s], r // S, "sums")
            yield from delay()
            assert loaded[s] == r
            read.append(r)
            empty[s].arrive()

    alive = [producer(True), producer(False), sums()] + [decoder(d) for d in range(4)] + \
            [issuer(q) for q in range(NI)]
    steps = 0
    while alive:
        steps += 1
        assert steps < 100000, f"no progress (seed {seed})"
        for e in list(landing):
            e[0] -= 1
            if e[0] <= 0:
                landing.remove(e)
                e[1].arrive()
        rnd.shuffle(alive)
        for co in list(alive):
            if rnd.random() < 0.3:
                continue
            try:
                next(co)
            except StopIteration:
                alive.remove(co)
    assert sorted(mma) == read == list(range(len(rounds)))


@pytest.mark.parametrize("S,NI", [(6, 2), (4, 2)])
def test_ring_with_the_sums_warp_is_exact(S, NI):
    for seed in range(150):
        run(seed, S, NI)
