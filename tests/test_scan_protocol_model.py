"""A host-side model of kernels whose roles talk through mbarriers polled by parity (no GPU).

A parity poll is only sound while the barrier is at most one phase ahead of the waiter: two phases ahead it blocks for good,
three ahead it passes on stale data.  The model runs a protocol (ring indices, parities, arrival counts) as a discrete-event
simulation under random and extreme role speeds, decides every wait by the parity rule alone, and checks against the true phase
counts that no wait is ever lapped, that none passes early, and that every role finishes.  The protocols themselves, with
variants that must be reported, are in test_scan_protocol_int8.py, test_scan_protocol_f16.py and test_state_protocol.py; the tests
here show that the model reports each kind of mistake.
"""
import heapq
import random

import pytest


class Bar:
    def __init__(self, name, count):
        self.name, self.count, self.pending, self.completed = name, count, count, 0

    def arrive(self, k=1):
        for _ in range(k):
            self.pending -= 1
            assert self.pending >= 0, f"{self.name}: more arrivals than the count of a phase"
            if self.pending == 0:
                self.completed += 1
                self.pending = self.count

    def poll(self, parity, want):
        """Hardware rule: true iff the phase of that parity has completed.  `want` is the number of
        completed phases the waiter really needs (model-side truth, for the checks only)."""
        assert self.completed <= want, f"{self.name}: lapped (completed {self.completed}, waiter needs {want})"
        ok = (self.completed & 1) != parity
        assert ok == (self.completed >= want), f"{self.name}: parity rule and phase count disagree"
        return ok


class Sim:
    """Roles are generators yielding ('wait', bar, parity, want) | ('work', t) | ('arrive', bar, k)
    | ('async', t, [(bar, k), ...]) (arrivals that happen t later: a TMA load landing, an MMA commit)."""

    def __init__(self, seed):
        self.rng = random.Random(seed)
        self.now = 0.0
        self.events = []   # (time, seq, kind, payload)
        self.seq = 0
        self.blocked = {}  # role name -> (gen, wait tuple)
        self.live = 0

    def push(self, t, kind, payload):
        self.seq += 1
        heapq.heappush(self.events, (t, self.seq, kind, payload))

    def spawn(self, name, gen):
        self.live += 1
        self.push(0.0, "run", (name, gen))

    def step_role(self, name, gen):
        while True:
            try:
                op = next(gen)
            except StopIteration:
                self.live -= 1
                return
            if op[0] == "work":
                self.push(self.now + op[1], "run", (name, gen))
                return
            if op[0] == "arrive":
                op[1].arrive(op[2])
                self.wake()
            elif op[0] == "async":
                self.push(self.now + op[1], "arrivals", op[2])
            elif op[0] == "wait":
                if not op[1].poll(op[2], op[3]):
                    self.blocked[name] = (gen, op)
                    return

    def wake(self):
        for name in list(self.blocked):
            gen, op = self.blocked[name]
            if op[1].poll(op[2], op[3]):
                del self.blocked[name]
                self.push(self.now, "run", (name, gen))

    def run(self):
        while self.events:
            self.now, _, kind, payload = heapq.heappop(self.events)
            if kind == "run":
                self.step_role(*payload)
            else:
                for bar, k in payload:
                    bar.arrive(k)
                self.wake()
        assert self.live == 0 and not self.blocked, f"deadlock: blocked {sorted(self.blocked)}"


def _run(producer, consumer, count=1):
    sim = Sim(0)
    full, free = Bar("FULL", count), Bar("FREE", 1)
    sim.spawn("producer", producer(full, free))
    sim.spawn("consumer", consumer(full, free))
    sim.run()


def _produce(n, respect_free=True):
    def gen(full, free):
        for i in range(n):
            if respect_free:
                yield ("wait", free, (i & 1) ^ 1, i)
            yield ("async", 1.0, [(full, 1)])
            yield ("work", 1.0)
    return gen


def _consume(n, work=3.0, skip=0):
    def gen(full, free):
        for i in range(skip, n):
            yield ("wait", full, i & 1, i + 1)
            yield ("work", work)
            yield ("arrive", free, 1)
    return gen


def test_a_sound_handshake_passes():
    _run(_produce(9), _consume(9))


def test_a_lapped_wait_is_reported():
    with pytest.raises(AssertionError, match="lapped"):
        _run(_produce(9, respect_free=False), _consume(9))


def test_a_wait_that_passes_early_is_reported():
    with pytest.raises(AssertionError, match="disagree"):
        _run(_produce(9), _consume(9, skip=1))   # (a fresh barrier answers the parity of phase 1 with yes)


def test_a_missing_arrival_is_reported():
    with pytest.raises(AssertionError, match="deadlock"):
        _run(_produce(9), _consume(9), count=2)
