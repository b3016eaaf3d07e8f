"""The GEMM's barriers on a model of its roles (gemm.cu), run in many orders.

A wait names a phase by its parity alone, so a role that lets a barrier run two
phases ahead of it waits for ever.  On the GPU such a fault shows only when one
role is late by chance; here the roles are Python generators, and the scheduler
holds any of them back for as long as another can go on."""
import itertools
import random

import pytest

from test_kernel_order import kernel_text


class Bar:
    """An mbarrier: `count` arrivals complete a phase."""

    def __init__(self, count):
        self.count, self.pending, self.phase = count, count, 0

    def arrive(self):
        self.pending -= 1
        if self.pending == 0:
            self.pending = self.count
            self.phase += 1

    def passed(self, parity):  # the phase of this parity has completed
        return (self.phase & 1) != parity


def roles(steps, xs, ws, nb, missed):
    """Generators of producer, issuer, tensor core and the four dequantising
    groups over items of `steps[i]` two-k-block steps; each yields the
    conditions it waits for.  missed: the producer looks at the step of xs steps
    ago only, however soon its A stage comes round again."""
    joint = xs == 4 and not missed
    full_x = [Bar(1) for _ in range(xs)]
    full_w, empty_w = [Bar(1) for _ in range(ws)], [Bar(2) for _ in range(ws)]
    full_a, empty = [Bar(1) for _ in range(4)], [Bar(1) for _ in range(4)]
    done, acc_free = [Bar(1) for _ in range(nb)], [Bar(4) for _ in range(nb)]
    queue = []  # the barriers that the MMAs issued so far complete, in order
    pad = [(n + 1) & ~1 for n in steps]
    first = [sum(pad[:i]) for i in range(len(steps))]

    def producer():
        w = x = 0
        hist, used = [], [0] * 4  # the issued steps' A stages and parities
        numbers, seen = [], 0
        sx, usedx = 0, [0] * xs

        def put_w():
            nonlocal w
            yield lambda: empty_w[w % ws].passed((w // ws & 1) ^ 1)
            full_w[w % ws].arrive()
            w += 1

        for i, n in enumerate(steps):
            nw = pad[i] // 2
            yield from put_w()
            for p in range(n):
                if p % 2 == 0 and p // 2 + 1 < nw:
                    yield from put_w()
                number = first[i] + p
                if joint:
                    yield lambda: empty[sx].passed(usedx[sx] ^ 1)
                else:
                    ahead = xs
                    if number - 4 in numbers and not missed:
                        ahead = min(xs, sum(m >= number - 4 for m in numbers))
                    while x - seen >= ahead:
                        yield lambda: empty[hist[seen][0]].passed(hist[seen][1])
                        seen += 1
                full_x[sx].arrive()
                usedx[sx] ^= 1
                sx = (sx + 1) % xs
                numbers.append(number)
                hist.append((number & 3, used[number & 3]))
                used[number & 3] ^= 1
                x += 1
            if joint and n & 1:
                sx = (sx + 1) % xs

    def issuer():
        x, used = 0, [0] * 4
        for i, n in enumerate(steps):
            yield lambda: acc_free[i % nb].passed((i // nb & 1) ^ 1)
            for p in range(n):
                s = (first[i] + p) & 3
                yield lambda: full_a[s].passed(used[s])
                if joint:
                    yield lambda: full_x[s].passed(used[s])
                else:
                    yield lambda: full_x[x % xs].passed(x // xs & 1)
                used[s] ^= 1
                queue.append((empty[s],))
                x += 1
            queue.append((done[i % nb],))
        queue.append(None)

    def tensor_core():
        at = 0
        while True:
            yield lambda: at < len(queue)
            if queue[at] is None:
                return
            for b in queue[at]:
                b.arrive()
            at += 1

    def group(g):
        used = 0

        def step(i, p):
            nonlocal used
            t = (first[i] + p) >> 1
            yield lambda: full_w[t % ws].passed(t // ws & 1)
            if p < steps[i]:
                yield lambda: empty[g].passed(used ^ 1)
                used ^= 1
                full_a[g].arrive()
            # (of a tile's two halves the group holds one: two groups release it)
            empty_w[t % ws].arrive()

        begun = False
        for i in range(len(steps)):
            for p in range(((g - first[i]) & 3) + (4 if begun else 0), pad[i], 4):
                yield from step(i, p)
            begun = False
            if i + 1 < len(steps):  # one step of the next item before this one's epilogue
                p = (g - first[i + 1]) & 3
                if p < pad[i + 1]:
                    yield from step(i + 1, p)
                    begun = True
            yield lambda: done[i % nb].passed(i // nb & 1)
            acc_free[i % nb].arrive()

    return [producer(), issuer(), tensor_core()] + [group(g) for g in range(4)]


def finishes(gens, pick):
    """Runs the roles, pick(ready) choosing the next among those that can go on."""
    waits = {}
    for i, g in enumerate(gens):
        waits[i] = next(g, None)
    waits = {i: c for i, c in waits.items() if c is not None}
    while waits:
        ready = [i for i, c in waits.items() if c()]
        if not ready:
            return False
        i = pick(ready)
        c = next(gens[i], None)
        if c is None:
            del waits[i]
        else:
            waits[i] = c
    return True


SHAPES = [(4, 4, 2), (3, 2, 1)]  # activation stages, code tiles, accumulators: BN <= 128 and 256
STEPS = [1, 2, 3, 4, 5, 6, 9, 16]


def all_finish(steps, shape, missed):
    orders = list(itertools.permutations(range(7)))
    rng = random.Random(str((steps, shape)))
    for order in rng.sample(orders, 60) + [(1, 2, 3, 4, 5, 6, 0)]:  # the last: a late producer
        rank = {r: i for i, r in enumerate(order)}
        if not finishes(roles(steps, *shape, missed), lambda ready: min(ready, key=rank.get)):
            return False
    return all(finishes(roles(steps, *shape, missed), rng.choice) for _ in range(20))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n", STEPS)
def test_every_order_finishes(n, shape):
    assert all_finish([n] * 7, shape, False)
    assert all_finish([n, 3, n, n, 1, 2, n], shape, False)
    assert all_finish([1, 1, n, 1, n, n, 5], shape, False)


def test_the_model_sees_a_missed_phase():
    # an odd item leaves a step number out, and its A stage is used again before a
    # late producer has looked
    assert not all_finish([3] * 7, SHAPES[0], True)
    assert not all_finish([1] * 7, SHAPES[1], True)
    assert all_finish([4] * 7, SHAPES[0], True)


def test_the_kernel_looks_as_the_model_does():
    body = kernel_text("gemm.cu", "gemm_kernel")
    assert "mbar_wait(&empty[sx], ((usedx >> sx) & 1u) ^ 1u, abort)" in body
    assert "const int ahead = (near & 8u) ? min(XS, __popc(near)) : XS;" in body
    assert "for (; xn - seen >= ahead && ok; ++seen)" in body
