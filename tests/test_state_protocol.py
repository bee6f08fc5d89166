"""The handshake of the fused state kernel (csrc/chunk_state_pass.cu) on the host-side model of test_scan_protocol_model.py:
the loading warp with its ring of LUT_state, the ring of slabs, the warps that re-quantise (the state warps themselves or two of their
own), the issuing warp, the state warps.  Every wait is decided by parity alone and checked against the true phase counts.  A second
model lets arrivals go missing and waits run out: every role must still come to its end.  `broken` names variants that the models
must report."""
import heapq

import pytest

from test_scan_protocol_model import Bar, Sim


class Named:
    """A hardware barrier of a fixed number of warps: arrivals beyond a phase count towards the next, nothing runs out."""

    def __init__(self, warps):
        self.warps, self.here, self.waiting = warps, 0, []


class StateSim(Sim):
    """With hardware barriers: ("hw_arrive", barrier) and ("hw_sync", barrier), one warp each."""

    def hw(self, barrier, wake):
        barrier.here += 1
        if wake is not None:
            barrier.waiting.append(wake)
        if barrier.here == barrier.warps:
            barrier.here = 0
            for w in barrier.waiting:
                self.push(self.now, "run", w)
            barrier.waiting = []

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
                self.issue(op)
            elif op[0] == "hw_arrive":
                self.hw(op[1], None)
            elif op[0] == "hw_sync":
                self.hw(op[1], (name, gen))
                return
            elif not self.passes(name, gen, op):
                return

    def issue(self, op):
        self.push(self.now + op[1], "arrivals", op[2])

    def passes(self, name, gen, op):
        ok = op[1].poll(op[2], op[3])
        if not ok:
            self.blocked[name] = (gen, op)
        return ok


def build(sim, chunks, speed, few, na, slabs=None, broken=None):
    """few: the eight state warps re-quantise, one chunk ahead, behind a ring of six; else two row warps behind a ring of four.
    na accumulators.  slabs: live slabs of every chunk (of up to four; drawn if not given).  broken: a variant that the model must
    report."""
    rng = sim.rng
    slots, rows = (6, 8) if few else (4, 2)
    bars = lambda name, n, count: [Bar(f"{name}{i}", count) for i in range(n)]
    # (FULL: the loading warp's own arrival, and the copies' bytes)
    fulls, ready, freed = bars("FULL", slots, 2), bars("READY", slots, rows), bars("FREE", slots, 1)
    accs, acc_free, luts = bars("ACC", na, 1), bars("ACC_FREE", na, 8), bars("LUT", 4, 1)
    meet = Named(8)
    most = max(slabs) if slabs else rng.choice([1, 2, 4])   # slabs of a chunk
    slabs = slabs or [rng.randint(1, most) for _ in range(chunks)]
    whole = few and chunks * most <= slots                  # the ring holds the call
    if few:
        slabs = [most if k == 0 or whole else n for k, n in enumerate(slabs)]
    first = [sum(slabs[:k]) for k in range(chunks)]
    last_of = {first[k] + slabs[k] - 1 for k in range(chunks)}
    t = lambda role: rng.expovariate(1.0) * speed[role]
    full = lambda ring, i, lost: ("wait", ring[i % len(ring)], i // len(ring) & 1, i // len(ring) + 1, lost)
    free = lambda ring, i, lost: ("wait", ring[i % len(ring)], (i // len(ring) & 1) ^ 1, i // len(ring), lost)

    def loader():
        lost = []   # filled when a wait gives up: the role ends
        known = 1 if few else 0   # chunk from which on LUT_state decides what is loaded
        ahead = 6 if broken == "LUT_state six chunks ahead" else 4
        copy = lambda i: ("async", t("load"), [(fulls[i % slots], 1)])

        def fetch(k):
            if known <= k < chunks and not whole:
                yield ("async", t("load"), [(luts[(k - known) % 4], 1)])

        if few:
            for i in range(sum(slabs) if whole else slabs[0]):
                yield ("arrive", fulls[i % slots], 1)
                yield copy(i)
        else:
            yield from fetch(0)
            yield copy(0)
        for k in range(1, known + ahead):
            yield from fetch(k)
        for k in range(chunks if whole else known, chunks):
            yield full(luts, k - known, lost)
            if lost:
                return
            for i in range(first[k], first[k] + slabs[k]):
                if broken != "slabs without FREE":
                    yield free(freed, i, lost)
                if lost:
                    return
                yield ("arrive", fulls[i % slots], 1)
                if few or i > 0:
                    yield copy(i)
            yield from fetch(k + ahead)

    def issuer():
        lost = []
        for k in range(chunks):
            for i in range(first[k], first[k] + slabs[k]):
                yield full(ready, i, lost)
                if lost:
                    return
                if i == first[k] and broken != "accumulator without ACC_FREE":
                    yield free(acc_free, k, [])   # (gives up, goes on)
                yield ("work", t("mma") * 0.2)
                yield ("async", t("mma"), [(freed[i % slots], 1)] + ([(accs[k % na], 1)] if i in last_of else []))

    def quantise(at, lost):   # from slab at[0] on to the last of its chunk; where a wait gives up the next call goes on with that slab
        while True:
            i = at[0]
            yield full(fulls, i, lost)
            if lost:
                return
            if broken == "slabs ready twice":
                yield ("arrive", ready[i % slots], 1)
            yield ("work", t("rows"))
            yield ("arrive", ready[i % slots], 1)
            at[0] += 1
            if i in last_of:
                return

    def row_warp():
        lost, at = [], [0]
        for _ in range(chunks):
            yield from quantise(at, lost)
            if lost:
                return

    def state_warp(w):
        at = [0]
        for k in range(chunks):
            for _ in range((k == 0) + (k + 1 < chunks) if few else 0):
                yield from quantise(at, [])
            yield ("work", t("state"))
            if w == 0:
                gone = []
                yield full(accs, k, gone)
                if gone and broken == "the warp that polls for the MMAs leaves":
                    return
            yield ("hw_sync", meet)
            yield ("work", t("state"))
            yield ("arrive", acc_free[k % na], 1)

    sim.spawn("load", loader())
    sim.spawn("issue", issuer())
    for w in range(0 if few else rows):
        sim.spawn(f"row{w}", row_warp())
    for w in range(8):
        sim.spawn(f"state{w}", state_warp(w))


ROLES = ("load", "rows", "mma", "state")


FORMS = [(True, 1), (True, 2), (False, 1), (False, 2)]


@pytest.mark.parametrize("few,na", FORMS)
@pytest.mark.parametrize("chunks", [1, 2, 3, 4, 5, 8, 33])
def test_every_wait_is_sound_at_random_and_extreme_speeds(chunks, few, na):
    for seed in range(24):
        sim = StateSim(seed)
        speed = {r: 10.0 ** sim.rng.uniform(-2, 2) for r in ROLES}
        if seed < len(ROLES):
            speed = {r: 100.0 if r == ROLES[seed] else 0.01 for r in ROLES}
        build(sim, chunks, speed, few, na, slabs=[4] * chunks if seed % 3 == 0 else None)
        sim.run()


class LossySim(StateSim):
    """Asynchronous arrivals (loads and MMAs that never complete) are dropped, the `drop`-th and with `rest` all after it;
    waits give up after a while."""

    PATIENCE = 50.0

    def __init__(self, seed, drop, rest):
        super().__init__(seed)
        self.drop, self.rest, self.gave_up = drop, rest, 0

    def issue(self, op):
        self.drop -= 1
        if self.drop > 0 or self.drop < 0 and not self.rest:
            super().issue(op)

    def passes(self, name, gen, op):
        if (op[1].completed & 1) != op[2]:
            return True
        self.blocked[name] = (gen, op)
        self.push(self.now + self.PATIENCE, "expire", (name, op))
        return False

    def wake(self):
        for name in list(self.blocked):
            gen, op = self.blocked[name]
            if (op[1].completed & 1) != op[2]:
                del self.blocked[name]
                self.push(self.now, "run", (name, gen))

    def run(self):
        while self.events:
            self.now, _, kind, payload = heapq.heappop(self.events)
            if kind == "run":
                self.step_role(*payload)
            elif kind == "expire":
                name, op = payload
                if name in self.blocked and self.blocked[name][1] is op:
                    self.gave_up += 1
                    if len(op) > 4:
                        op[4].append(True)
                    self.push(self.now, "run", (name, self.blocked.pop(name)[0]))
            else:
                for bar, k in payload:
                    bar.arrive(k)
                self.wake()
        return self.live == 0


SPEED = dict(load=1.0, rows=1.0, mma=0.3, state=1.0)


@pytest.mark.parametrize("rest", [False, True])
@pytest.mark.parametrize("few,na", FORMS)
@pytest.mark.parametrize("chunks", [1, 2, 3, 5])
def test_every_role_ends_when_arrivals_go_missing(chunks, few, na, rest):
    gave_up = 0
    for drop in range(1, 6 * chunks):
        sim = LossySim(drop, drop, rest)
        build(sim, chunks, SPEED, few, na)
        assert sim.run(), drop
        gave_up += sim.gave_up
    assert gave_up > 0


@pytest.mark.parametrize("broken,barrier,few", [("LUT_state six chunks ahead", "LUT", True), ("LUT_state six chunks ahead", "LUT", False),
                                                ("slabs without FREE", "F", True), ("slabs without FREE", "F", False),
                                                ("accumulator without ACC_FREE", "ACC", True), ("accumulator without ACC_FREE", "ACC", False),
                                                ("slabs ready twice", "READY", True), ("slabs ready twice", "READY", False)])
def test_broken_variants_are_reported(broken, barrier, few):
    reported = 0
    for seed in range(24):
        sim = StateSim(seed)
        speed = {r: 100.0 if r == ROLES[seed % len(ROLES)] else 0.01 for r in ROLES}
        build(sim, 33, speed, few, 1, slabs=[4] * 33, broken=broken)
        try:
            sim.run()
        except AssertionError as e:
            reported += barrier in str(e)
    assert reported > 0


def test_a_state_warp_that_leaves_would_not_let_the_others_end():
    # the warp that polls for the MMAs comes to the barrier of the eight also where it has given up; if it left the others would stay there
    stuck = 0
    for drop in range(1, 20):
        sim = LossySim(drop, drop, rest=True)
        build(sim, 5, SPEED, True, 1, broken="the warp that polls for the MMAs leaves")
        stuck += not sim.run()
    assert stuck > 0
