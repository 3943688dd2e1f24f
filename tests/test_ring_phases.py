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


def tma_ring(steps_of_tiles, slots, pairs, singles, bufs, partner_frees):
    """codec_umma.cuh, and pass 1 of codec_umma_roundtrip.cuh: one load per stage, `pairs` operands whose two issuers take
    alternate stages of a tile and `singles` with one, an accumulator per issuer; partner_frees: the issuer whose turn it is
    not frees the stage as well."""
    ops = pairs + singles
    r = Ring(slots, 1, ops + (pairs if partner_frees else 0), bufs, 2 * pairs + singles, 1)

    def issuer(op, half, halves):
        step = 0
        for tile, nst in enumerate(steps_of_tiles):
            yield r.acc_empty[tile % bufs], 1 - tile // bufs % 2
            for st in range(nst):
                slot = step % slots
                yield r.full[slot], step // slots % 2
                if halves == 1 or st % 2 == half:
                    r.consume("rows", slot, step)
                    r.later(("mma", op, half), lambda slot=slot, step=step: free(slot, step))
                elif partner_frees:
                    free(slot, step)
                step += 1
                yield None
            r.later(("mma", op, half), lambda buf=tile % bufs: r.acc_full[buf].arrive())

    def free(slot, step):
        r.consume("rows", slot, step)
        if r.empty[slot].pending == 1:
            r.release(slot, ("rows",))
        r.empty[slot].arrive()

    def epilogue():
        for tile in range(len(steps_of_tiles)):
            yield r.acc_full[tile % bufs], tile // bufs % 2
            r.acc_empty[tile % bufs].arrive()

    r.roles = [_producer(r, "rows", sum(steps_of_tiles), True), epilogue()]
    r.roles += [issuer(op, half, 2) for op in range(pairs) for half in (0, 1)] + [issuer(pairs + op, 0, 1) for op in range(singles)]
    return r


@pytest.mark.parametrize("pairs,singles,bufs", [(1, 0, 2), (1, 1, 2), (2, 0, 2), (2, 0, 1), (0, 3, 1)])
def test_tma_projection(pairs, singles, bufs):
    for slots in (2, 4, 5, 10):
        for tiles in ((1,), (1, 1, 1), (8, 4), (7, 7, 7, 3), (16, 16, 8)):
            for seed in range(60):
                tma_ring(tiles, slots, pairs, singles, bufs, partner_frees=True).run(random.Random(seed))


def test_a_stage_its_reader_alone_frees_can_pass_by_the_partner():
    with pytest.raises(AssertionError):
        for seed in range(300):
            tma_ring((16, 16, 8), 5, 1, 0, 2, partner_frees=False).run(random.Random(seed))
