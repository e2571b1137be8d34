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
_CONST = dict(re.findall(r"constexpr int (kThreads|kTabThreads) = (\d+);", open(SOURCE).read()))
N_COMPUTE, N_TAB = int(_CONST["kThreads"]) // 32, int(_CONST["kTabThreads"]) // 32


class Stuck(Exception):
    pass


class Twice(Exception):
    pass


class Cta:
    """Warps are generators of operations: ("arrive" | "sync", barrier), ("wait", event) -> whether it came in time, ("until", n):
    the storing warp has taken n output tiles."""

    def __init__(self, rng, n_c, so, short, lost, old):
        self.rng, self.n_c, self.so, self.short, self.lost, self.old = rng, n_c, so, short, lost, old
        self.size = {4: N_COMPUTE + 1 + N_TAB, 5: N_COMPUTE + 1, 6: N_COMPUTE + 1, 1: N_COMPUTE, 3: N_TAB}
        self.size.update({8 + q: N_COMPUTE // 4 for q in range(4)})
        self.count = {b: [] for b in self.size}   # warps of the present generation
        self.done, self.coming, self.fail, self.taken = set(), set(), False, 0

    def signal(self, *event):  # a load or a product: it completes some time later, or never
        if event not in self.lost:
            self.coming.add(event)

    def compute(self, w):
        n_c, so = self.n_c, self.so
        gave_up, c = 0, 0
        yield "arrive", 4
        while c < n_c:
            gave_up = 1
            if not so and not (yield "wait", ("pre", c)):
                break
            if not (yield "wait", ("d1", c)):
                break
            if not so:
                yield "sync", 8 + w % 4
            yield "arrive", 5
            gave_up = 2
            if not so:
                if c >= 1 and not (yield "wait", ("stg", c - 1)):
                    break
                if not (yield "wait", ("o2", c)):
                    break
                yield "arrive", 6
            gave_up = 3
            if not (yield "wait", ("g2", c)):
                break
            yield "arrive", 4
            if self.short and c == n_c - 1:
                yield "sync", 1
            gave_up = 0
            c += 1
        if gave_up and self.old:
            yield "arrive", 4
            yield "arrive", 5
            yield "arrive", 6
        elif gave_up:
            while c < n_c:
                if gave_up < 2:
                    if not so:
                        yield "sync", 8 + w % 4
                    yield "sync", 5
                if not so and gave_up < 3:
                    yield "until", c
                    yield "sync", 6
                if c + 1 < n_c:
                    yield "sync", 4
                if self.short and c == n_c - 1:
                    yield "sync", 1
                c, gave_up = c + 1, 1

    def tabler(self, w):
        for c in range(self.n_c):
            if self.old and self.fail:
                break
            if c + 1 < self.n_c:
                yield "sync", 3
            yield "wait", ("full", c)
            yield "sync", 4

    def producer(self, w):
        for c in range(min(2, self.n_c)):
            self.signal("full", c)
        for c in range(self.n_c):
            if self.old and self.fail:
                break
            if not self.so:
                yield "sync", 6
                self.taken = c + 1
            if not self.fail:
                if c + 2 < self.n_c and (yield "wait", ("g2", c)) and not self.fail:
                    self.signal("full", c + 2)
                self.signal("stg", c)

    def issuer(self, w):
        def pre(c):
            yield "wait", ("full", c)
            if not self.fail:
                self.signal("pre", c)
        for c in range(self.n_c):
            if self.old and self.fail:
                break
            yield "sync", 4
            if c == 0:
                yield from pre(0)
            if not self.fail:
                self.signal("d1", c)
            yield "sync", 5
            if not self.fail:
                self.signal("o2", c)
                self.signal("g2", c)
            if c + 1 < self.n_c:
                yield from pre(c + 1)
        if self.old and self.fail:
            yield "arrive", 4

    def run(self):
        kinds = [self.compute] * N_COMPUTE + [self.issuer, self.producer] + [self.tabler] * N_TAB
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
            ready = [i for i in pending if i not in asleep and (pending[i][0] != "wait" or pending[i][1] in self.done)
                     and (pending[i][0] != "until" or self.taken >= pending[i][1])]
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
                if kind in ("wait", "until"):
                    step(i, True)
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
    return [set()] + [{(e, c)} for c in range(n_c) for e in ("full", "d1", "g2") + (() if so else ("pre", "o2", "stg"))]


@pytest.mark.parametrize("so,short", [(False, False), (False, True), (True, False)])
def test_every_warp_leaves_whatever_runs_out(so, short):
    for n_c in (1, 2, 4):
        for lost, seed in itertools.product(_lost(n_c, so), range(40)):
            Cta(random.Random(seed), n_c, so, short, lost, old=False).run()


def test_the_model_sees_warps_that_leave_early():
    """Waiters that leave as soon as they see the failure, and compute warps that arrive once on every hand-off before they leave:
    the counts can no longer come out, and somebody stays behind."""
    stuck = 0
    for seed in range(40):
        try:
            Cta(random.Random(seed), 3, False, False, {("full", 1)}, old=True).run()
        except Stuck:
            stuck += 1
    assert stuck > 0
