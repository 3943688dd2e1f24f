"""The stage rings of the kernels whose MMA issuers take turns, as a model on the CPU: roles as coroutines, barriers that tell
a waiting role no more than the parity of their phase, and schedules that hold a role up for as long as they like.  No role may
read or overwrite a stage at the wrong time, nor wait for a phase that has gone by."""

import os
import random
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_13332_b200", "csrc")


def _constant(file, name):
    return int(re.search(rf"\b{name} = (\d+)[;,]", open(os.path.join(CSRC, file)).read()).group(1))


class Barrier:
    def __init__(self, count):
        self.count = self.pending = count
        self.phase = 0

    def arrive(self):
        self.pending -= 1
        if self.pending == 0:
            self.pending, self.phase = self.count, self.phase + 1

    def passed(self, parity):
        return self.phase % 2 != parity


class Ring:
    """Roles yield (barrier, parity) to wait and None to let time pass; `later` runs what completes by itself, in order per key."""

    def __init__(self, slots, full, empty, bufs, acc_full, acc_empty):
        self.full, self.empty = [Barrier(full) for _ in range(slots)], [Barrier(empty) for _ in range(slots)]
        self.acc_full, self.acc_empty = [Barrier(acc_full) for _ in range(bufs)], [Barrier(acc_empty) for _ in range(bufs)]
        self.slots, self.bufs, self.holds, self.acc, self.queues, self.roles = slots, bufs, {}, {}, {}, []

    def later(self, key, action):
        self.queues.setdefault(key, []).append(action)

    def run(self, rng):
        waits, held, now = [None] * len(self.roles), {}, 0
        live = set(range(len(self.roles)))
        while live:
            now += 1
            if rng.random() < 0.02:                       # one role, or what it has under way, stands still for a while
                held[rng.choice([*live, *self.queues])] = now + rng.randint(50, 400)
            ready = [i for i in live if waits[i] is None or waits[i][0].passed(waits[i][1])]
            pending = [k for k, q in self.queues.items() if q]
            assert ready or pending, "every role waits for a phase that has gone by"
            free = [x for x in ready + pending if held.get(x, 0) <= now]
            if not free:
                now = min(held[x] for x in ready + pending)
                continue
            pick = rng.choice(free)
            if pick in self.queues:
                self.queues[pick].pop(0)()
                continue
            try:
                waits[pick] = next(self.roles[pick])
            except StopIteration:
                live.discard(pick)

    def fill(self, part, slot, step):
        assert (part, slot) not in self.holds, "a stage is overwritten before it has been consumed"
        self.holds[part, slot] = step
        self.full[slot].arrive()

    def consume(self, part, slot, step):
        assert self.holds.get((part, slot)) == step, "a stage is read that is not the one waited for"

    def release(self, slot, parts):
        for p in parts:
            del self.holds[p, slot]


def _producer(r, part, steps, asynchronous, first=0, stride=1):
    for step in range(first, steps, stride):
        slot, turn = step % r.slots, step // r.slots
        yield r.empty[slot], 1 - turn % 2
        if asynchronous:
            r.later(("load", part, slot), lambda slot=slot, step=step: r.fill(part, slot, step))
        else:
            r.fill(part, slot, step)
        yield None


def plain_ring(steps, slots, basis_warps, bufs, wait_all):
    """codec_plain_project.cuh: rows by TMA, a stage of the basis per warp in turn, two issuers in turn, sums per stage."""
    r = Ring(slots, 2, 1, bufs, 1, 1)

    def issuer(which):
        for step in range(steps):
            slot, buf = step % slots, step % bufs
            if step % 2 == which or wait_all:
                yield r.full[slot], step // slots % 2
            if step % 2 != which:
                continue
            yield r.acc_empty[buf], 1 - step // bufs % 2
            for part in ("rows", "basis"):
                r.consume(part, slot, step)

            def done(slot=slot, buf=buf, step=step):
                r.release(slot, ("rows", "basis"))
                r.empty[slot].arrive()
                r.acc[buf] = step
                r.acc_full[buf].arrive()
            r.later(("mma", which), done)
            yield None

    def sums():
        for step in range(steps):
            yield r.acc_full[step % bufs], step // bufs % 2
            assert r.acc[step % bufs] == step
            r.acc_empty[step % bufs].arrive()

    r.roles = [_producer(r, "rows", steps, True), issuer(0), issuer(1), sums()]
    r.roles += [_producer(r, "basis", steps, False, w, basis_warps) for w in range(basis_warps)]
    return r


@pytest.mark.parametrize("bufs", [2, 4])
@pytest.mark.parametrize("steps", [1, 7, 8, 41])
def test_plain_projection(steps, bufs):
    slots, basis = (_constant("codec_plain_project.cuh", n) for n in ("kStagesN", "kPlainBasisWarps"))
    for seed in range(150):
        plain_ring(steps, slots, basis, bufs, wait_all=False).run(random.Random(seed))


def test_an_issuer_that_looks_at_its_partners_stages_can_miss_one():
    with pytest.raises(AssertionError):
        for seed in range(150):
            plain_ring(41, 9, 4, 2, wait_all=True).run(random.Random(seed))
