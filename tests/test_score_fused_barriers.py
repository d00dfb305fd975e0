"""The barriers of the kernel for short bf16 prompts, walked on the CPU by its roles in any order (no GPU): no phase may pass a
waiting warp by, whose parity test would then miss it, and every role must come to its end."""
import os
import random
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_03409_b200", "csrc")
SLOTS = 8   # tiles in tensor memory
KEYS = 5    # key tiles in shared memory


def given_back():
    """From the source: arrivals that free a query stage, and whether the MMA warp that has not got the strip is one."""
    text = open(os.path.join(CSRC, "score_fused.cu")).read()
    products = text[text.index("---- products"):text.index("---- loads")]
    return int(re.search(r"bar_init\(q_empty \+ i, (\d+)\)", text).group(1)), "bar_arrive(q_empty" in products


class Barriers:
    def __init__(self):
        self.count, self.pending, self.done = {}, {}, {}

    def init(self, bar, count):
        self.count[bar] = self.pending[bar] = count
        self.done[bar] = 0

    def arrive(self, bar):
        self.pending[bar] -= 1
        if self.pending[bar] == 0:
            self.pending[bar] = self.count[bar]
            self.done[bar] += 1


def run(S, heads, stages, frees, other_frees, rng):
    """One CTA with `heads` heads of S strips; the roles as generators that yield what they wait for."""
    T = (S + 1) // 2
    b = Barriers()
    for i in range(stages):
        b.init(("q_full", i), 1)
        b.init(("q_empty", i), frees)
    for i in range(KEYS):
        b.init(("k_full", i), 1)
        b.init(("k_empty", i), 2)
    for i in range(SLOTS):
        b.init(("s_empty", i), 1)
        for odd in (0, 1):
            b.init(("s_full", odd, i), 1)
    issued = [0, 0]            # the MMA warps' progress
    pipe = [[], []]            # an MMA warp's commits, which arrive in order, some time later

    def full(kind, n, ring):   # completion n // ring of the barrier
        return (kind, n % ring), n // ring

    def loader():
        def load(kind, n, ring):
            if n >= ring:
                yield (kind + "_empty", n % ring), n // ring - 1
            b.arrive((kind + "_full", n % ring))
        nq = nk = 0
        strips = heads * S
        def q():
            nonlocal nq
            if nq < strips:
                yield from load("q", nq, stages)
                nq += 1
        yield from q()
        for _ in range(T):
            yield from load("k", nk, KEYS)
            nk += 1
        for _ in range(stages - 1):
            yield from q()
        for i in range(heads):
            for s in reversed(range(S)):
                yield from q()
                if s % 2 == 0 and i + 1 < heads:
                    yield from load("k", nk, KEYS)
                    nk += 1

    def products(odd):
        strip = tile = key0 = 0
        for _ in range(heads):
            for s in reversed(range(S)):
                top = s // 2
                yield full("q_full", strip, stages)
                if s % 2 == odd:
                    for at, g in enumerate(reversed(range(top + 1))):
                        n, k = tile + at, key0 + T - 1 - g
                        if s >= S - 2:
                            yield full("k_full", k, KEYS)
                        while issued[1 - odd] <= n - SLOTS:
                            yield None
                        if n >= SLOTS:
                            yield ("s_empty", n % SLOTS), n // SLOTS - 1
                        pipe[odd].append([("s_full", odd, n % SLOTS)] + [("k_empty", k % KEYS)] * (g == top) +
                                         [("q_empty", strip % stages)] * (g == 0))
                    after = (s - 1) // 2 + 1 if s > 0 else 0 if (S - 1) % 2 == odd else (S - 1) // 2 + 1
                    issued[odd] = tile + top + 1 + after
                else:
                    if other_frees:
                        b.arrive(("q_empty", strip % stages))
                    if s == S - 1 and odd:
                        yield full("k_full", key0, KEYS)
                        b.arrive(("k_empty", key0 % KEYS))
                        issued[odd] = tile + top + 1
                tile += top + 1
                strip += 1
            key0 += T

    def retire(odd):
        while True:
            if pipe[odd]:
                for bar in pipe[odd].pop(0):
                    b.arrive(bar)
            yield None

    def readers(team):
        tile, uses = 0, [0] * SLOTS
        for _ in range(heads):
            for s in reversed(range(S)):
                n = s // 2 + 1
                if s % 2 == team:
                    for x in range(n):
                        yield ("s_full", team, (tile + x) % SLOTS), uses[(tile + x) % SLOTS]
                        uses[(tile + x) % SLOTS] += 1
                    for x in reversed(range(n)):
                        yield None
                        b.arrive(("s_empty", (tile + x) % SLOTS))
                tile += n

    roles = [loader(), products(0), products(1), readers(0), readers(1), retire(0), retire(1)]
    waits = [None] * len(roles)
    left = set(range(5))
    weight = [rng.choice([0.01, 0.1, 1.0]) for _ in roles]
    idle = 0
    while left:
        if rng.random() < 0.01:
            weight = [rng.choice([0.01, 0.1, 1.0]) for _ in roles]
        r = rng.choices(range(len(roles)), weight)[0]
        if r < 5 and r not in left:
            continue
        if waits[r] is not None:
            bar, want = waits[r]
            if b.done[bar] > want + 1:
                return "%s passed by" % (bar,)
            if b.done[bar] < want:  # (the parity of the phase before last would let it through)
                return "%s waited for too early" % (bar,)
            if b.done[bar] == want:
                idle += 1
                if idle > 50000:
                    return "stuck"
                continue
        idle = 0 if r < 5 else idle + 1
        if idle > 50000:
            return "stuck"
        try:
            waits[r] = next(roles[r])
        except StopIteration:
            left.discard(r)
    return None


@pytest.mark.parametrize("stages", [3, 6])
@pytest.mark.parametrize("S", range(1, 11))
def test_no_phase_passes_unseen(S, stages):
    frees, other_frees = given_back()
    rng = random.Random(S * 100 + stages)
    for _ in range(12):
        assert run(S, 9 if S < 4 else 4, stages, frees, other_frees, rng) is None


def test_the_walk_shows_a_stage_given_back_by_one_warp_alone():
    rng = random.Random(1)
    assert any(run(1, 9, 3, 1, False, rng) == "('q_full', %d) passed by" % i for _ in range(40) for i in range(3))
