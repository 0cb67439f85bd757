"""Host model of the CTA pairs' ring in the code product (fq_tc.cu, tc_pair_kernel): two CTAs, a producer
of activation tiles and D decoders of W warps in each, one MMA issuer in rank 0.  A parity wait only
tells a phase from the one before it, and a decoder waits for a stage only in every D-th round, so the
model checks at every poll that the parity says exactly whether the awaited phase is complete, that
every stage holds its round's data when the MMAs read it, and that all rounds finish, under random
interleavings."""
import random

import pytest


class Barrier:
    def __init__(self, count):
        self.count, self.pending, self.phase = count, count, 0

    def arrive(self):
        self.pending -= 1
        if self.pending == 0:
            self.pending, self.phase = self.count, self.phase + 1

    def passed(self, k):
        """A parity wait for phase k (-1: before the first)."""
        by_parity = (self.phase & 1) != (k & 1)
        assert by_parity == (self.phase > k), f"phase {self.phase}, waiting for {k}"
        return by_parity


def _run(S, D, W, rounds, seed):
    rng = random.Random(seed)
    # full: the leader's arrival, both CTAs' bytes, every decoder warp of both; empty: the MMAs' commit
    full = [Barrier(1 + 2 + 2 * W) for _ in range(S)]
    empty = [[Barrier(1) for _ in range(S)] for _ in range(2)]
    a = [[[None] * W for _ in range(S)] for _ in range(2)]     # round held by each warp's rows of A
    b = [[None] * S for _ in range(2)]
    in_flight = []                                             # MMAs issued, completed in order

    def producer(rank):
        for i in range(rounds):
            s = i % S
            while not empty[rank][s].passed(i // S - 1):
                yield
            if rank == 0:
                full[s].arrive()
            yield
            b[rank][s] = i
            full[s].arrive()
            yield

    def decoder(rank, d, w):
        for i in range(d, rounds, D):
            s = i % S
            while not empty[rank][s].passed(i // S - 1):
                yield
            a[rank][s][w] = i
            yield
            full[s].arrive()
            yield

    def issuer():
        for i in range(rounds):
            s = i % S
            while not full[s].passed(i // S):
                yield
            in_flight.append(i)
            yield

    def tensor_core():
        for i in range(rounds):
            while not in_flight or in_flight[0] != i:
                yield
            s = i % S
            for rank in range(2):
                assert a[rank][s] == [i] * W and b[rank][s] == i
                empty[rank][s].arrive()
            in_flight.pop(0)
            yield

    tasks = [producer(r) for r in range(2)] + [issuer(), tensor_core()]
    tasks += [decoder(r, d, w) for r in range(2) for d in range(D) for w in range(W)]
    weight = [rng.choice((1, 1, 1, 8)) for _ in tasks]         # some roles run far ahead
    for _ in range(4000 * rounds):
        if not tasks:
            return
        j = rng.choices(range(len(tasks)), weight)[0]
        if next(tasks[j], "done") == "done":
            del tasks[j], weight[j]
    assert not tasks, "rounds left"


@pytest.mark.parametrize("S,D,W", [(6, 6, 2), (9, 9, 1), (7, 6, 2)])
@pytest.mark.parametrize("rounds", [1, 5, 9, 14, 71])
def test_waits_are_exact_and_data_in_place(S, D, W, rounds):
    assert D <= S
    for seed in range(6):
        _run(S, D, W, rounds, seed)


def test_the_model_sees_a_ring_shorter_than_its_decoders():
    """With more decoders than stages a decoder can fall two phases behind: the check must fail."""
    with pytest.raises(AssertionError):
        for seed in range(200):
            _run(3, 7, 1, 60, seed)
