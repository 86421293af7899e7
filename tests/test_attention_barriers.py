"""The order that the self-attention kernel's barriers give, on a model of its
warps (loads, the two issuing streams, the two softmax streams): every product
reads the blocks that it is meant to read, however long each load takes.  The
ring depths, and what a stream without a block waits for, are the kernel's own,
read from its source."""
import heapq
import os
import random
import re

import pytest

SRC = open(os.path.join(os.path.dirname(os.path.abspath(__file__)), os.pardir,
                        "paper_2608_29809_gb300", "csrc", "attention_tc.cu")).read()
# a stream without a block in a unit waits for the O of the unit before
EMPTY_WAITS = bool(re.search(r"if \(i0 >= n\) \{[^}]*mbar_sleep\(o_free", SRC))
KS, VS = (int(re.search(rf"{n}_STAGES = (\d+);", SRC).group(1)) for n in "KV")


class Bar:
    """mbarrier: a wait on a parity passes when the phase in progress has the
    other one."""

    def __init__(self, count=1):
        self.count = self.left = count
        self.phase = 0

    def arrive(self):
        self.left -= 1
        if self.left == 0:
            self.phase, self.left = self.phase + 1, self.count


class Fault(Exception):
    pass


def simulate(units, ks, vs, seed, empty_waits=EMPTY_WAITS):
    """Runs one CTA's units, (tiles, key blocks) each; raises Fault."""
    rng = random.Random(seed)
    now, heap, serial = 0.0, [], 0

    def at(t, fn):
        nonlocal serial
        serial += 1
        heapq.heappush(heap, (t, serial, fn))

    def latency():  # now and then a load takes far longer than its neighbours
        return rng.uniform(1, 3) if rng.random() < 0.9 else rng.uniform(20, 300)

    bars = lambda n, count=1: [Bar(count) for _ in range(n)]  # noqa: E731
    q_full, q_empty, o_full, o_free, meet = Bar(), Bar(2), Bar(2), Bar(2), Bar(2)
    k_full, k_empty, v_full, v_empty = bars(ks), bars(ks, 2), bars(vs), bars(vs, 2)
    s_full, p_ready, pv_done = ([bars(2), bars(2)] for _ in range(3))
    held = {"K": [None] * ks, "V": [None] * vs}
    products, o_read = [0] * len(units), [0] * len(units)
    pipe = 0.0

    def load(what, stage, block, full):
        def land():
            held[what][stage] = block
            full.arrive()
        at(now + latency(), land)

    def loads_k():
        g = 0
        for uc, (_, n) in enumerate(units):
            yield q_empty, (uc & 1) ^ 1
            at(now + latency(), q_full.arrive)
            for _ in range(n):
                yield k_empty[g % ks], ((g // ks) & 1) ^ 1
                load("K", g % ks, g, k_full[g % ks])
                g += 1
                yield rng.uniform(0, 1)

    def loads_v():
        for g in range(sum(n for _, n in units)):
            yield v_empty[g % vs], ((g // vs) & 1) ^ 1
            load("V", g % vs, g, v_full[g % vs])
            yield rng.uniform(0, 1)

    def product(what, stage, block, then):
        """An MMA and the commits behind it: in order, done a little later."""
        nonlocal pipe
        pipe = max(pipe, now) + rng.uniform(0.1, 1)

        def done():
            if held[what][stage] != block:
                raise Fault(f"{what} stage {stage}: block {held[what][stage]} for {block}")
            for b in then:
                b.arrive()
        if held[what][stage] != block:
            raise Fault(f"{what} stage {stage}: block {held[what][stage]} for {block}")
        at(pipe, done)

    def issuer(x):
        g0 = ns = np = 0
        for uc, (tiles, n) in enumerate(units):
            two = tiles == 2
            i0, di = (0, 1) if two else (x, 2)
            yield q_full, uc & 1
            i_s = i0
            for i in range(i0, n, di):
                while i_s < n and i_s < i + 2 * di:
                    g, b = g0 + i_s, ns & 1
                    yield k_full[g % ks], (g // ks) & 1
                    yield pv_done[x][b], ((ns >> 1) & 1) ^ 1
                    then = [s_full[x][b]] + [k_empty[g % ks]] * (1 if two else 2)
                    product("K", g % ks, g, then + ([q_empty] if i_s + di >= n else []))
                    i_s, ns = i_s + di, ns + 1
                g, b = g0 + i, np & 1
                if i == i0:
                    yield o_free, (uc & 1) ^ 1
                    if uc and o_read[uc - 1] != 2:
                        raise Fault(f"unit {uc} writes O before unit {uc - 1}'s was read")
                yield v_full[g % vs], (g // vs) & 1
                yield p_ready[x][b], (np >> 1) & 1
                np += 1
                then = [pv_done[x][b]] + [v_empty[g % vs]] * (1 if two else 2)
                product("V", g % vs, g, then + ([o_full] if i + di >= n else []))
                products[uc] += 1
            if i0 >= n:
                at(max(pipe, now), q_empty.arrive)
                if empty_waits:
                    yield o_free, (uc & 1) ^ 1
                at(max(pipe, now), o_full.arrive)
            g0 += n

    def softmax(x):
        cnt = met = 0
        for uc, (tiles, n) in enumerate(units):
            two = tiles == 2
            for _ in range(0 if two else x, n, 1 if two else 2):
                yield s_full[x][cnt & 1], (cnt >> 1) & 1
                yield rng.uniform(0, 3)
                p_ready[x][cnt & 1].arrive()
                cnt += 1
            if not two:
                meet.arrive()
                yield meet, met
                met ^= 1
            yield o_full, uc & 1
            if products[uc] != n * tiles:
                raise Fault(f"unit {uc}: O read after {products[uc]} of {n * tiles} products")
            yield rng.uniform(0, 3)
            o_read[uc] += 1
            o_free.arrive()

    waiting = []
    ready = [loads_k(), loads_v(), issuer(0), issuer(1), softmax(0), softmax(1)]
    while True:
        while ready:
            actor = ready.pop(rng.randrange(len(ready)))
            step = next(actor, None)
            if isinstance(step, tuple):
                waiting.append((actor, *step))
            elif step is not None:
                at(now + step, lambda a=actor: ready.append(a))
            passed = [w for w in waiting if (w[1].phase & 1) != w[2]]
            waiting = [w for w in waiting if (w[1].phase & 1) == w[2]]
            ready += [w[0] for w in passed]
        if not heap:
            break
        now, _, fn = heapq.heappop(heap)
        fn()
        passed = [w for w in waiting if (w[1].phase & 1) != w[2]]
        waiting = [w for w in waiting if (w[1].phase & 1) == w[2]]
        ready += [w[0] for w in passed]
    if waiting:
        raise Fault("a wait never ends")


UNITS = {
    "one tile": [(1, 52)] * 3,
    "one tile, odd": [(1, 13), (1, 7), (1, 31), (1, 3), (1, 2)],
    "two tiles": [(2, 13), (2, 6), (2, 2)],
    "both": [(2, 13), (1, 13), (2, 5), (1, 8), (1, 21), (2, 2), (1, 17)],
    "single blocks": [(1, 9), (1, 1), (1, 1), (2, 4), (1, 1), (2, 1), (1, 1), (1, 2), (1, 1)],
}


@pytest.mark.parametrize("units", UNITS)
def test_products_read_the_blocks_they_are_meant_to(units):
    for seed in range(120):
        simulate(UNITS[units], KS, VS, seed)


@pytest.mark.parametrize("ks,vs", [(6, 7), (5, 8)])
def test_the_model_sees_rings_of_odd_depth(ks, vs):
    """With one tile a unit the streams take the blocks in turn, so an odd ring
    hands a stage to the other stream each time round."""
    with pytest.raises(Fault):
        for seed in range(400):
            simulate(UNITS["one tile"], ks, vs, seed)


def test_the_model_sees_a_stream_without_a_block_that_does_not_wait():
    with pytest.raises(Fault):
        for seed in range(400):
            simulate(UNITS["single blocks"], KS, VS, seed, empty_waits=False)
