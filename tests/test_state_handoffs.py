"""The hand-offs between the warps of the state-passing kernel, as a model on the CPU: every warp is the sequence of barrier
operations that it has in `chunk_state.cu`, a scheduler runs them in random orders, and any bounded wait may run out at any time.
Whatever runs out where, every warp has to reach the end, and none may be counted twice in one generation of a hardware barrier
(it would complete early, and what is left could never complete it again)."""
import itertools
import os
import random
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_06034_b200", "csrc", "chunk_state.cu")
_CONST = dict(re.findall(r"constexpr int (kChain|kAux|kThreads|kTabThreads) = (\d+);", open(SOURCE).read()))
N_CHAIN, N_AUX, N_TAB = (int(_CONST[k]) // 32 for k in ("kChain", "kAux", "kTabThreads"))
RING = 3  # K, Q tiles


class Stuck(Exception):
    pass


class Twice(Exception):
    pass


class Cta:
    """Warps are generators of operations: ("arrive" | "sync", barrier), ("wait", event) -> whether it came in time, ("count", event):
    one of the arrivals that complete an event."""

    def __init__(self, rng, n_c, so, short, lost, old):
        self.rng, self.n_c, self.so, self.short, self.lost, self.old = rng, n_c, so, short, lost, old
        self.size = {4: N_CHAIN + 1 + N_TAB, 5: N_CHAIN + 1, 6: N_CHAIN + 1, 7: N_AUX + 1, 8: N_AUX + 1, 1: N_AUX, 3: N_TAB}
        self.needs = {"nrm": N_AUX, "tab": N_TAB, "ost": N_AUX}
        self.count = {b: [] for b in self.size}   # warps of the present generation
        self.arrived = {}
        self.done, self.coming, self.fail = set(), set(), False

    def signal(self, *event):  # a load or a product: it completes some time later, or never
        if event not in self.lost:
            self.coming.add(event)

    def chain(self, w):
        n_c = self.n_c
        taken, good = 0, True

        def prefetch(c):
            return (yield "wait", ("tab", c)) and (yield "wait", ("u", c))
        for hand in (4, 6):
            yield "arrive", hand
            taken += 1
        good = yield from prefetch(0)
        c = 0
        while good and c < n_c:
            good = yield "wait", ("d1", c)
            if not good:
                break
            yield "arrive", 5
            taken += 1
            if c + 1 < n_c:
                good = yield from prefetch(c + 1)
                for half, hand in enumerate((4, 6)):
                    if good:
                        good = yield "wait", ("su%d" % half, c)
                    if good:
                        yield "arrive", hand
                        taken += 1
            else:
                good = yield "wait", ("su1", c)
            c += 1
        if not good and self.old:
            for hand in (4, 5, 6):
                yield "arrive", hand
        elif not good:
            for i in range(taken, 3 * n_c):
                yield "sync", (4, 6, 5)[i % 3]

    def aux(self, w):
        n_c, so = self.n_c, self.so
        taken = 0

        def norms(c):
            if c >= n_c:
                return True
            if so and w >= N_CHAIN + N_AUX // 2:
                yield "count", ("nrm", c)
                return True
            if not (yield "wait", ("kq", c)):
                return False
            yield "count", ("nrm", c)
            return True
        good = yield from norms(0)
        if so:
            c = 1
            while good and c < n_c:
                good = c < 2 or (yield "wait", ("tab", c - 2))
                good = good and (yield from norms(c))
                c += 1
            return
        yield "sync", 1
        c = 0
        while good and c < n_c:
            good = yield "wait", ("pt", c)
            if good:
                yield "arrive", 7
                taken += 1
                good = c > 0 or (yield from norms(1))
                good = good and (yield from norms(c + 2))
            if good:
                good = yield "wait", ("o2", c)
            if good and c + 1 < n_c:
                yield "arrive", 8
                taken += 1
            if good and c >= 2:
                good = yield "wait", ("stg", c - 2)
            if good:
                yield "count", ("ost", c)
            c += 1
        if not good and self.old:
            yield "arrive", 7
            yield "arrive", 8
        elif not good:
            for i in range(taken, 2 * n_c - 1):
                yield "sync", (7, 8)[i % 2]

    def tabler(self, w):
        for c in range(self.n_c):
            if self.old and self.fail:
                break
            yield "sync", 3
            yield "wait", ("nrm", c)
            yield "count", ("tab", c)
            yield "wait", ("kq", c)
            yield "wait", ("w", c)
            yield "sync", 4

    def producer(self, w):
        n_c = self.n_c
        asked = set()

        def load(what, c):
            assert (what, c) not in asked
            # the barrier's phase before is complete: an arrival on it twice in one phase is a fault of the GPU
            before = c - (RING if what == "kq" else 2)
            assert before < 0 or (what, before) in self.done, (what, c)
            if c < n_c:
                asked.add((what, c))
                self.signal(what, c)
        for c in range(RING):
            load("kq", c)
            if c < 2:
                load("w", c)
                load("u", c)
        for c in range(n_c):
            if self.fail:
                break
            if c + 2 < n_c:
                if not (yield "wait", ("d1", c)) or self.fail:
                    break
                load("w", c + 2)
                if c > 0:
                    load("u", c + 2)
                if not (yield "wait", ("su1", c)) or self.fail:
                    break
                if c == 0:
                    load("u", 2)
                load("kq", c + 3)
            if not self.so:
                if not (yield "wait", ("ost", c)) or self.fail:
                    break
                self.signal("stg", c)

    def issuer(self, w):
        for c in range(self.n_c):
            if self.old and self.fail:
                break
            yield "sync", 4
            yield "sync", 6
            if not self.fail:
                self.signal("d1", c)
            if not self.so:
                if c > 0:
                    yield "sync", 8
                if not self.fail:
                    self.signal("pt", c)
            yield "sync", 5
            if not self.fail:
                self.signal("su0", c)
                self.signal("su1", c)
            if not self.so:
                yield "sync", 7
                if not self.fail:
                    self.signal("o2", c)

    def run(self):
        kinds = [self.chain] * N_CHAIN + [self.aux] * N_AUX + [self.issuer, self.producer] + [self.tabler] * N_TAB
        warps = [k(i) for i, k in enumerate(kinds)]
        frozen = self.rng.choice([-1, *range(len(warps))])  # runs when nothing else can, until a wait has run out
        early = self.rng.choice((0.0, 0.002))  # how often a wait runs out though something could still go on
        pending = {}  # warp -> operation it stands at
        asleep = {}   # warp -> barrier it waits on

        def step(i, value=None):
            try:
                pending[i] = warps[i].send(value)
            except StopIteration:
                pending.pop(i, None)

        for i in range(len(warps)):
            step(i)
        while pending:
            ready = [i for i in pending if i not in asleep and (pending[i][0] != "wait" or pending[i][1] in self.done)]
            waiting = [i for i in pending if pending[i][0] == "wait" and pending[i][1] not in self.done]
            awake = [i for i in ready if i != frozen or self.fail]
            if self.coming and (self.rng.random() < 0.3 or not awake):
                self.done.add(self.coming.pop())
            elif waiting and (not awake or self.rng.random() < (0.1 if self.fail else early)):
                self.fail = True
                step(self.rng.choice(waiting), False)
            elif ready:
                i = self.rng.choice(awake or ready)
                kind, what = pending[i]
                if kind == "wait":
                    step(i, True)
                    continue
                if kind == "count":
                    self.arrived[what] = self.arrived.get(what, 0) + 1
                    if self.arrived[what] == self.needs[what[0]] and what not in self.lost:
                        self.done.add(what)
                    step(i)
                    continue
                here = self.count[what]
                if i in here and not self.old:
                    raise Twice((i, what))
                here.append(i)
                if kind == "sync":
                    asleep[i] = what
                full = len(here) == self.size[what]
                woken = [j for j in here if asleep.get(j) == what] if full else []
                if full:
                    here.clear()
                for j in woken:
                    del asleep[j]
                    step(j)
                if kind == "arrive":
                    step(i)
            else:
                raise Stuck({i: pending[i] for i in pending})


def _lost(n_c, so):
    """No event lost, and every single one of each kind in turn."""
    return [set()] + [{(e, c)} for c in range(n_c) for e in ("kq", "w", "u", "d1", "su0", "su1", "nrm", "tab") + (() if so else ("pt", "o2", "ost", "stg"))]


@pytest.mark.parametrize("so,short", [(False, False), (False, True), (True, False)])
def test_every_warp_leaves_whatever_runs_out(so, short):
    for n_c in (1, 2, 4):
        for lost, seed in itertools.product(_lost(n_c, so), range(40 if n_c < 4 else 12)):
            Cta(random.Random(seed), n_c, so, short, lost, old=False).run()


def test_the_model_sees_warps_that_leave_early():
    """Waiters that leave as soon as they see the failure, and compute warps that arrive once on every hand-off before they leave:
    the counts can no longer come out, and somebody stays behind."""
    stuck = 0
    for seed in range(40):
        try:
            Cta(random.Random(seed), 3, False, False, {("kq", 1)}, old=True).run()
        except Stuck:
            stuck += 1
    assert stuck > 0
