"""The hand-offs between the warps of the state-passing kernel, as a model on the CPU: every warp is the sequence of barrier
operations that it has in `chunk_state.cu`, a scheduler runs them in random orders, and any bounded wait may run out at any time.
Whatever runs out where, every warp has to reach the end, and none may be counted twice in one generation of a hardware barrier
(it would complete early, and what is left could never complete it again). A wait on an mbarrier asks for the parity of a phase:
no warp, however slow, may still stand before its wait on a phase when the next phase of that barrier is complete too (the parity
would read "not complete"), and nobody may arrive on a barrier before the phase that the arrival is meant for."""
import itertools
import os
import random
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_06034_b200", "csrc", "chunk_state.cu")
_CONST = dict(re.findall(r"constexpr int (kChain|kAux|kThreads|kTabThreads) = (\d+);", open(SOURCE).read()))
N_CHAIN, N_AUX, N_TAB = (int(_CONST[k]) // 32 for k in ("kChain", "kAux", "kTabThreads"))
RING = int(re.search(r"constexpr int kRing = (\d+);", open(SOURCE).read()).group(1))  # K, Q tiles
# phases of every event that its barriers tell apart: chunk c is on barrier c mod this (kq .. stg as the kernel declares them)
SLOTS = {name: RING if size == "kRing" else int(size or 1)
         for line in re.findall(r"__shared__ uint64_t (bar_.*?);", open(SOURCE).read())
         for name, size in re.findall(r"bar_(\w+)(?:\[(\w+)\])?", line)}


class Stuck(Exception):
    pass


class Twice(Exception):
    pass


class Overtaken(Exception):
    pass


class WrongPhase(Exception):
    pass


class Cta:
    """Warps are generators of operations: ("arrive" | "sync", barrier), ("wait", event) -> whether it came in time, ("count", event):
    one of the arrivals that complete an event. An event (name, chunk) is a phase of barrier chunk mod SLOTS[name]. `slow`: warps
    that take a step only when nobody else can; without `lost` events no wait runs out then."""

    def __init__(self, rng, n_c, so, nrm, lost=(), old=False, slow=None, slots=SLOTS):
        self.rng, self.n_c, self.so, self.nrm, self.lost, self.old, self.slow, self.slots = rng, n_c, so, nrm, lost, old, slow, slots
        self.size = {4: N_CHAIN + 1 + N_TAB, 5: N_CHAIN + 1, 6: N_CHAIN + 1, 7: N_AUX + 1, 8: N_AUX + 1, 1: N_AUX, 3: N_TAB}
        self.needs = {"nrm": N_AUX, "tab": N_TAB, "ost": N_AUX}
        self.count = {b: [] for b in self.size}   # warps of the present generation
        self.arrived = {}
        self.phases, self.fail = {}, False         # barrier -> phases that are complete
        self.loads, self.products = [], []         # on their way: loads in any order, products in the order they were issued

    def barrier(self, name, c):
        n = self.slots[name]
        return (name, c % n), c // n

    def signal(self, name, c):  # a load, a product or a store: it completes some time later, or never
        bar, phase = self.barrier(name, c)
        if self.phases.get(bar, 0) != phase and not self.fail:
            raise WrongPhase((name, c))
        if (name, c) not in self.lost:
            (self.loads if name in ("kq", "w", "u", "stg") else self.products).append((name, c))

    def complete(self, name, c):
        bar, phase = self.barrier(name, c)
        if self.phases.get(bar, 0) != phase and not self.fail:
            raise WrongPhase((name, c))
        self.phases[bar] = max(self.phases.get(bar, 0), phase + 1)

    def come(self, name, c):
        bar, phase = self.barrier(name, c)
        if self.phases.get(bar, 0) > phase + 1 and not self.fail:
            raise Overtaken((name, c))
        return self.phases.get(bar, 0) > phase

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
            if c >= n_c or not self.nrm:
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
            while good and self.nrm and c < n_c:
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
            if self.nrm:
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
        patient = self.slow is not None
        # slow warps run when nothing else can; of those that the test does not name, until a wait has run out
        slow = self.slow if patient else {self.rng.choice([-1, *range(len(warps))])}
        early = 0.0 if patient else self.rng.choice((0.0, 0.002))  # how often a wait runs out though something could still go on
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
            ready = [i for i in pending if i not in asleep and (pending[i][0] != "wait" or self.come(*pending[i][1]))]
            waiting = [i for i in pending if pending[i][0] == "wait" and not self.come(*pending[i][1])]
            awake = [i for i in ready if i not in slow or (self.fail and not patient)]
            if (self.loads or self.products) and (self.rng.random() < 0.3 or not awake):
                if self.loads and (not self.products or self.rng.random() < 0.5):
                    self.complete(*self.loads.pop(self.rng.randrange(len(self.loads))))
                else:
                    self.complete(*self.products.pop(0))
            elif waiting and not (patient and ready) and (not awake or self.rng.random() < (0.1 if self.fail else early)):
                self.fail = True
                step(self.rng.choice(waiting), False)
            elif ready:
                i = self.rng.choice(awake or ready)
                kind, what = pending[i]
                if kind == "wait":
                    step(i, True)
                    continue
                if kind == "count":
                    bar, phase = self.barrier(*what)
                    if self.phases.get(bar, 0) != phase and not self.fail:
                        raise WrongPhase(what)
                    self.arrived[what] = self.arrived.get(what, 0) + 1
                    if self.arrived[what] == self.needs[what[0]] and what not in self.lost:
                        self.complete(*what)
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


def _lost(n_c, so, nrm):
    """No event lost, and every single one of each kind in turn."""
    kinds = ("kq", "w", "u", "d1", "su0", "su1", "tab") + (("nrm",) if nrm else ()) + (() if so else ("pt", "o2", "ost", "stg"))
    return [set()] + [{(e, c)} for c in range(n_c) for e in kinds]


@pytest.mark.parametrize("so,nrm", [(False, True), (False, False), (True, True), (True, False)])
def test_every_warp_leaves_whatever_runs_out(so, nrm):
    for n_c in (1, 2, 4):
        for lost, seed in itertools.product(_lost(n_c, so, nrm), range(40)):
            Cta(random.Random(seed), n_c, so, nrm, lost).run()


def test_the_model_sees_warps_that_leave_early():
    """Waiters that leave as soon as they see the failure, and compute warps that arrive once on every hand-off before they leave:
    the counts can no longer come out, and somebody stays behind."""
    stuck = 0
    for seed in range(40):
        try:
            Cta(random.Random(seed), 3, False, True, {("kq", 1)}, old=True).run()
        except Stuck:
            stuck += 1
    assert stuck > 0


WARPS = N_CHAIN + N_AUX + 2 + N_TAB
# one warp of each part, and the ones of a part that do something of their own (norms of K, norms of Q)
SLOW = [{0}, {N_CHAIN}, {N_CHAIN + N_AUX - 1}, {WARPS - N_TAB - 2}, {WARPS - N_TAB - 1}, {WARPS - 1}, {WARPS - N_TAB - 1, 0},
        {WARPS - N_TAB - 1, N_CHAIN}, {WARPS - N_TAB - 1, WARPS - 1}, set()]


@pytest.mark.parametrize("so,nrm", [(False, True), (False, False), (True, True), (True, False)])
def test_no_phase_is_lost_however_slow_a_warp_is(so, nrm):
    """Nothing is lost and nothing runs out; the slow warps stay behind as far as the others can go without them. More chunks than twice
    the longest ring."""
    for slow, seed in itertools.product(SLOW, range(6)):
        cta = Cta(random.Random(seed), 9, so, nrm, slow=slow)
        cta.run()
        assert not cta.fail


@pytest.mark.parametrize("so,nrm", [(False, True), (False, False), (True, True), (True, False)])
def test_the_model_sees_a_phase_that_is_overtaken(so, nrm):
    """Two barriers for the state update's completion: the loading warp is two chunks behind before anybody needs what it asks for."""
    with pytest.raises(Overtaken):
        for seed in range(6):
            Cta(random.Random(seed), 9, so, nrm, slow={WARPS - N_TAB - 1}, slots={**SLOTS, "su0": 2, "su1": 2}).run()
