"""The handshake of the fused state kernel (csrc/chunk_state_pass.cu) on the host-side model of test_scan_protocol_model.py:
the loading warp, the ring of slabs, the warps that re-quantise (the state warps themselves or two of their own), the issuing warp,
the state warps.  Every wait is decided by parity alone and checked against the true phase counts.  A second model lets arrivals
go missing and waits run out: every role must still come to its end."""
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


def build(sim, chunks, speed, few, na, slabs=None):
    """few: the eight state warps re-quantise, one chunk ahead, behind a ring of six; else two row warps behind a ring of four.
    na accumulators.  slabs: live slabs of every chunk (of up to four; drawn if not given)."""
    rng = sim.rng
    slots, rows = (6, 8) if few else (4, 2)
    bars = lambda name, n, count: [Bar(f"{name}{i}", count) for i in range(n)]
    fulls, ready, freed = bars("FULL", slots, 1), bars("READY", slots, rows), bars("FREE", slots, 1)
    accs, acc_free = bars("ACC", na, 1), bars("ACC_FREE", na, 8)
    meet = Named(8)
    slabs = slabs or [rng.randint(1, 4) for _ in range(chunks)]
    first = [sum(slabs[:k]) for k in range(chunks)]
    t = lambda role: rng.expovariate(1.0) * speed[role]
    full = lambda ring, i, lost: ("wait", ring[i % len(ring)], i // len(ring) & 1, i // len(ring) + 1, lost)
    free = lambda ring, i, lost: ("wait", ring[i % len(ring)], (i // len(ring) & 1) ^ 1, i // len(ring), lost)

    def loader():
        lost = []   # filled when a wait gives up: the role ends
        for i in range(sum(slabs)):
            yield free(freed, i, lost)
            if lost:
                return
            yield ("async", t("load"), [(fulls[i % slots], 1)])

    def issuer():
        lost = []
        for k in range(chunks):
            for i in range(first[k], first[k] + slabs[k]):
                yield full(ready, i, lost)
                if lost:
                    return
                if i == first[k]:
                    yield free(acc_free, k, [])   # (gives up, goes on)
                yield ("work", t("mma") * 0.2)
                last = i + 1 == first[k] + slabs[k]
                yield ("async", t("mma"), [(freed[i % slots], 1)] + ([(accs[k % na], 1)] if last else []))

    def quantise(k, lost):
        for i in range(first[k], first[k] + slabs[k]):
            yield full(fulls, i, lost)
            if lost:
                return
            yield ("work", t("rows"))
            yield ("arrive", ready[i % slots], 1)

    def row_warp():
        lost = []
        for k in range(chunks):
            yield from quantise(k, lost)
            if lost:
                return

    def state_warp(w):
        lost = []
        if few:
            yield from quantise(0, lost)
        for k in range(chunks):
            if few and k + 1 < chunks and not lost:
                yield from quantise(k + 1, lost)
            yield ("work", t("state"))
            if w == 0:
                yield full(accs, k, [])
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
