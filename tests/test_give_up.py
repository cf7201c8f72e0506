"""Who decides that a solve ends early (CPU).  The warps of a CTA meet at named
barriers, which have no limit: if each warp took its own decision when a wait runs
out, those that go on would be left there.  A model of the persistent engine's CTA
-- producer, eight compute warps in two groups that take turns, publisher -- under
every order of events: with the producer alone deciding, every run ends; with a
limit at each warp's waits some run does not.  And the engine's source is held to
the first."""
import os
import random
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2403_18619_gb300",
                    "csrc")
WARPS, GROUP = 8, 4


class Cta:
    """Events of one CTA; a wait is a condition on them."""

    def __init__(self, rng, each_warp):
        self.rng, self.each_warp = rng, each_warp
        self.tasks = [rng.choice(["turn", "panel", "pivot"]) for _ in range(rng.randint(2, 7))]
        self.handed = []            # descriptors: a task's kind, or "stop"
        self.taken = []             # warps that have read each descriptor
        self.issued = self.landed = 0
        self.released = []          # warps that have left each copy's buffer
        self.done = []              # warps that have finished each task
        self.published = 0
        self.arrived = {"cta": 0, 0: 0, 1: 0}   # barrier -> arrivals ever

    def wait(self, condition):
        """A wait of a compute warp: False if it runs out (own limit)."""
        while not condition():
            if self.each_warp and self.rng.random() < 0.01:
                return False
            yield
        return True

    def barrier(self, name, arrive_only=False):
        phase = self.arrived[name] // WARPS
        self.arrived[name] += 1
        while not arrive_only and self.arrived[name] // WARPS == phase:
            yield

    def producer(self):
        for kind in self.tasks + ["stop"]:
            if kind != "stop" and self.rng.random() < 0.08:
                kind = "stop"  # the inputs' wait has run out, or another CTA's has
            i = len(self.handed)
            while i >= 2 and self.taken[i - 2] < WARPS:
                yield
            self.handed.append(kind)
            self.taken.append(0)
            self.done.append(0)
            yield
            if kind == "stop":
                break
            if kind != "pivot":
                while self.issued >= 2 and self.released[self.issued - 2] < WARPS:
                    yield
                self.released.append(0)
                self.issued += 1
            else:
                while self.published <= i:
                    yield

    def copies(self):
        while True:
            if self.landed < self.issued:
                self.landed += 1
            yield "idle"

    def publisher(self):
        i = 0
        while True:
            while len(self.handed) <= i:
                yield
            if self.handed[i] == "stop":
                return
            while self.done[i] < WARPS:
                yield
            self.published += 1
            i += 1

    def warp(self, w):
        g, copy = w // GROUP, 0
        if g == 1:
            yield from self.barrier(0, arrive_only=True)
        for i in range(len(self.tasks) + 1):
            if not (yield from self.wait(lambda: len(self.handed) > i)):
                return
            kind = self.handed[i]
            self.taken[i] += 1
            if kind == "stop":
                return
            if kind != "pivot":
                if not (yield from self.wait(lambda: self.landed > copy)):
                    return
            if kind == "turn":
                yield from self.barrier(g)
                yield
                yield from self.barrier(1 - g, arrive_only=True)
            else:
                yield from self.barrier("cta")
                yield from self.barrier("cta")
            if kind != "pivot":
                self.released[copy] += 1
                copy += 1
            self.done[i] += 1

    def run(self):
        """Random order of events; whether every warp has left in the end."""
        actors = [self.producer(), self.publisher()] + [self.warp(w) for w in range(WARPS)]
        memory = self.copies()
        for _ in range(20000):
            if not actors:
                return True
            a = self.rng.choice(actors + [memory])
            try:
                next(a)
            except StopIteration:
                actors.remove(a)
        return False


@pytest.mark.parametrize("seed", range(60))
def test_every_run_ends_when_the_producer_decides(seed):
    assert Cta(random.Random(seed), each_warp=False).run()


def test_warps_deciding_for_themselves_do_not_all_end():
    assert not all(Cta(random.Random(s), each_warp=True).run() for s in range(40))


def test_only_the_producer_looks_at_the_limit_and_the_abort_flag():
    text = open(os.path.join(CSRC, "fw_ws.cuh")).read()
    bodies = {m.group(1): m.group(2) for m in
              re.finditer(r"^__device__[^;{}]*?(\w+)\((?:[^(){}]|\([^)]*\))*\) \{\n(.*?)^\}", text,
                          re.S | re.M)}
    assert {"mbar_wait", "wait_ge", "ws_engine"} <= set(bodies)
    reads = {n for n, b in bodies.items() if re.search(r"ld_\w+\(\s*[\w.>-]*abort_flag", b)}
    assert reads == {"wait_ge", "ws_engine"}
    claim = re.findall(r"ld_relaxed\(src\.abort_flag\)", bodies["ws_engine"])
    assert len(claim) == 1  # beside the claim of the next task
    limits = {n for n, b in bodies.items() if re.search(r"globaltimer\(\) - \w+", b)}
    assert limits == {"mbar_wait", "wait_ge"}
    # a phase of the CTA's own: no limit but for a copy that is lost
    assert "(uint64_t)timeout_ns + kLostNs" in bodies["mbar_wait"]
