"""CPU: the barriers of the prefill attention, stepped in random order.

A model of the roles of one CTA of prefill_attn_kernel (two producer warps, two issuing warps, eight
softmax warps) over the items of a run: which mbarrier each waits for and arrives on, in the order of
the kernel; copies and tensor-core work complete later, the products of a Q tile in their order.  An
mbarrier that is waited on by parity holds one phase nobody waited for yet: the model ends a run when a
barrier gets two phases ahead of a role that still has to see the first, when a wait lets a role go
before its phase is over, or when no role can go on.
Which tiles take a turn, and how many turns a group has behind it at its start, is asked of the
kernel's own header."""
import ctypes
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2505_20438_gb300", "csrc")
ITEMS_AHEAD, SOFT_WARPS = 4, 4


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("turns")
    src, lib = d / "turns.cpp", d / "turns.so"
    src.write_text('#include "ham_turns.cuh"\n'
                   'extern "C" int tiles(int nt0, int nt1) { return ham::turn_tiles(nt0, nt1); }\n'
                   'extern "C" unsigned before(int q) { return ham::turns_before(q); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)],
                   check=True)
    so = ctypes.CDLL(str(lib))

    def turns(q, tile, nt0, nt1):  # (takes, gives) in a tile of an item
        shared = tile < so.tiles(nt0, nt1)
        return shared, shared
    return turns, [so.before(0), so.before(1)]


def within_items(q, tile, nt0, nt1):
    """A rule the model has to refuse: Q tile 0 takes no turn in an item's first tile, Q tile 1 gives
    none in its last shared one, so that nothing orders the groups from one item to the next."""
    shared = nt0 if nt1 > 0 else 0
    return (tile < shared and (q == 1 or tile > 0),
            tile < (shared if q == 0 else shared - 1))


class Bar:
    def __init__(self, count):
        self.count = self.left = count
        self.phases = 0

    def arrive(self):
        self.left -= 1
        if self.left == 0:
            self.left, self.phases = self.count, self.phases + 1


class Cta:
    """One run.  Roles are generators that yield (barrier, phase) to wait for; phase n is the n-th
    completion, seen by the parity of n as the kernel sees it."""

    in_order = True  # a tile without products is released behind the products before it

    def __init__(self, items, rule, stages, tile_s, seed):
        (self.turns, self.before), self.items = rule, items
        self.rng, self.tile_s, self.stages = random.Random(seed), tile_s, stages
        self.full = [Bar(1) for _ in range(stages)]
        self.empty = [Bar(2) for _ in range(stages)]
        self.q_full, self.q_empty, self.o_full, self.pv_done = ([Bar(1), Bar(1)] for _ in range(4))
        self.s_full = [[Bar(1), Bar(1)] for _ in range(2)]
        self.p_full = [[Bar(SOFT_WARPS), Bar(SOFT_WARPS)] for _ in range(2)]
        self.turn = [Bar(SOFT_WARPS), Bar(SOFT_WARPS)]
        self.item_full = [Bar(1) for _ in range(ITEMS_AHEAD)]
        self.item_empty = [Bar(2 * SOFT_WARPS + 3) for _ in range(ITEMS_AHEAD)]
        self.pipes = [[] for _ in range(2)]  # commits of Q tile 0 / 1, completing in order
        self.copies = []                     # copies under way, completing in any order

    def item(self, k):
        yield self.item_full[k % ITEMS_AHEAD], k // ITEMS_AHEAD
        self.item_empty[k % ITEMS_AHEAD].arrive()

    def producer(self, is_v):
        e, q_issued = int(is_v), [0, 0]
        for k in range(len(self.items) + 1):
            if is_v:
                if k >= ITEMS_AHEAD:
                    yield self.item_empty[k % ITEMS_AHEAD], k // ITEMS_AHEAD - 1
                self.item_full[k % ITEMS_AHEAD].arrive()
            else:
                yield from self.item(k)
            if k == len(self.items):
                return
            nt0, nt1, _ = self.items[k]
            if is_v:
                for q in range(2 if nt1 else 1):
                    if q_issued[q]:
                        yield self.q_empty[q], q_issued[q] - 1
                    q_issued[q] += 1
                    self.copies.append(self.q_full[q])
            for _ in range(max(nt0, nt1)):
                if e >= self.stages:
                    yield self.empty[e % self.stages], e // self.stages - 1
                self.copies.append(self.full[e % self.stages])
                e += 2

    def blocks(self, q, k):
        nt0, nt1, odd = self.items[k]
        nt = nt1 if q else nt0
        return max(0, 2 * nt - (odd >> q & 1))

    def issuer(self, q):
        e, loads, parts, pipe = 0, 0, [0, 0], self.pipes[q]
        for k in range(len(self.items) + 1):
            yield from self.item(k)
            if k == len(self.items):
                return
            nt, nts, nb = self.items[k][q], max(self.items[k][:2]), self.blocks(q, k)
            e0, e = e, e + 2 * nts

            def entry(x):
                return self.full[x % self.stages], x // self.stages

            def scores(t):
                st, buf = (e0 + 2 * (t >> 1)) % self.stages, 0 if self.tile_s else t & 1
                pipe.append(self.s_full[q][buf])
                last = t + (2 if self.tile_s else 1) >= nb
                if self.tile_s or buf == 1 or last:
                    pipe.append(self.empty[st])
                if last:
                    pipe.append(self.q_empty[q])

            if nb:
                yield self.q_full[q], loads
                yield entry(e0)
                loads += 1
                scores(0)
                if not self.tile_s and nb > 1:
                    scores(1)
            for t in range(nb):
                buf, ev = t & 1, e0 + 2 * (t >> 1) + 1
                if buf == 0:
                    yield entry(ev)
                    if (t >> 1) + 1 < nt:
                        yield entry(ev + 1)
                yield self.p_full[q][buf], parts[buf]
                parts[buf] += 1
                pipe.append(self.pv_done[q])
                if t + 1 == nb:
                    pipe.append(self.o_full[q])
                if self.tile_s and buf == 1 and t + 1 < nb:
                    scores(t + 1)
                if not self.tile_s and t + 2 < nb:
                    scores(t + 2)
                if buf == 1 or t + 1 == nb:
                    pipe.append(self.empty[ev % self.stages])
            for x in range(e0 + 2 * nt, e):
                yield entry(x)
                if self.in_order:
                    pipe.append(self.empty[x % self.stages])
                else:
                    self.empty[x % self.stages].arrive()

    def softmax(self, q):
        seen, done, outs, turns = [0, 0], 0, 0, self.before[q]
        for k in range(len(self.items) + 1):
            yield from self.item(k)
            if k == len(self.items):
                return
            nt0, nt1, _ = self.items[k]
            nb = self.blocks(q, k)
            if nb == 0:
                continue
            for t in range(nb):
                buf = t & 1
                takes, gives = self.turns(q, t >> 1, nt0, nt1)
                if not self.tile_s or buf == 0:
                    s = 0 if self.tile_s else buf
                    yield self.s_full[q][s], seen[s]
                    seen[s] += 1
                    if self.tile_s and takes:
                        yield self.turn[q], turns - 2 * self.before[q]  # the parity of `turns`
                        turns += 1
                if t and self.rng.random() < 0.2:  # a raised maximum: O holds the block before
                    yield self.pv_done[q], done - 1
                if self.tile_s and gives and (buf == 1 or t + 1 == nb):
                    self.turn[q ^ 1].arrive()
                self.p_full[q][buf].arrive()
                done += 1
            yield self.o_full[q], outs
            outs += 1

    def run(self):
        """None if every role ends, else what is wrong."""
        roles = [self.producer(False), self.producer(True), self.issuer(0), self.issuer(1)]
        roles += [self.softmax(w // SOFT_WARPS) for w in range(2 * SOFT_WARPS)]
        weight = [self.rng.choice([1, 1, 3, 20]) for _ in roles]  # some are held up against others
        waits = [None] * len(roles)  # (barrier, phase); phase -1 is over when the CTA starts
        live = set(range(len(roles)))
        while live:
            if any(w is not None and w[0].phases > w[1] + 1 for w in waits):
                return "a barrier is two phases ahead of a wait"
            ready = [r for r in live if waits[r] is None or
                     (waits[r][0].phases & 1) != (waits[r][1] & 1)]
            late = [x for x in (0, 1) if self.pipes[x]]
            if not ready and not late and not self.copies:
                return "no role can go on"
            pick = self.rng.choices(["role", "pipe", "copy"],
                                    [3 * bool(ready), bool(late), bool(self.copies)])[0]
            if pick == "pipe":
                self.pipes[self.rng.choice(late)].pop(0).arrive()
            elif pick == "copy":
                self.copies.pop(self.rng.randrange(len(self.copies))).arrive()
            else:
                r = self.rng.choices(ready, [weight[x] for x in ready])[0]
                if waits[r] is not None and waits[r][0].phases < waits[r][1] + 1:
                    return "a wait ends before its phase"
                try:
                    waits[r] = next(roles[r])
                except StopIteration:
                    live.remove(r)
                    waits[r] = None
        return None


def _items(rng, kinds):
    return [(*rng.choice(kinds), rng.randrange(4)) for _ in range(rng.randint(3, 9))]


RUNS = [[(1, 1)], [(1, 2)], [(1, 0), (1, 1)], [(1, 1), (1, 2), (2, 2)], [(4, 5), (1, 1), (1, 2)],
        [(1, 0), (1, 2), (2, 3), (3, 3)], [(1, 0), (4, 5)], [(1, 0), (4, 0), (3, 3)]]


@pytest.mark.parametrize("kinds", RUNS)
@pytest.mark.parametrize("tile_s,stages", [(True, 5), (False, 10)])  # head_dim 128, 64
def test_every_wait_ends(rule, kinds, tile_s, stages):
    rng = random.Random(len(kinds))
    for seed in range(60):
        assert Cta(_items(rng, kinds), rule, stages, tile_s, seed).run() is None, f"run {seed}"


def test_turns_within_items_only_are_found_out():
    """The model sees the fault it is there for: turns that nothing carries from item to item."""
    rng = random.Random(7)
    wrong = {Cta(_items(rng, [(1, 1), (1, 2)]), (within_items, [0, 0]), 5, True, seed).run()
             for seed in range(200)}
    assert "a barrier is two phases ahead of a wait" in wrong


def test_releases_out_of_order_are_found_out(rule):
    """Stages of tiles that a Q tile does not reach, released ahead of the products before them: a
    producer can find a stage free that is still read."""
    rng = random.Random(1)
    wrong = set()
    for seed in range(400):
        cta = Cta(_items(rng, [(1, 0), (1, 2), (2, 3), (3, 3)]), rule, 5, True, seed)
        cta.in_order = False
        wrong.add(cta.run())
    assert "a wait ends before its phase" in wrong
