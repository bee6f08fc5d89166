"""The handshake of the fused state kernel (csrc/chunk_state_pass.cu) on the host-side model of test_scan_protocol_model.py:
three row warps, the warp that issues MMAs and loads, the state warps.  Every wait is decided by parity alone and checked against
the true phase counts.  A second model lets arrivals go missing and waits run out: every role must still come to its end.
`broken` is the form in which the row warps go on as if their waits had not given up."""
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


def build(sim, chunks, speed, broken=False):
    rng = sim.rng
    xfull, bfull, mma = [Bar("XFULL0", 1), Bar("XFULL1", 1)], Bar("BFULL", 1), Bar("MMA", 1)
    acc_free = Bar("ACC_FREE", 8)
    named = [Named(4), Named(4)]
    t = lambda role: rng.expovariate(1.0) * speed[role]
    full = lambda bar, use: ("wait", bar, use & 1, use + 1)
    free = lambda bar, use: ("wait", bar, (use & 1) ^ 1, use)

    def row_warp():
        lost = []   # filled when a wait gives up
        for k in range(chunks):
            if broken or not lost:
                yield (*full(xfull[k & 1], k >> 1), lost)
            if broken or not lost:
                yield ("work", t("rows"))
                yield ("hw_arrive", named[k & 1])
            else:
                yield ("hw_sync", named[k & 1])

    def issuer():
        yield ("async", t("load"), [(xfull[0], 1)])
        yield ("async", t("load"), [(bfull, 1)])
        if chunks > 1:
            yield ("async", t("load"), [(xfull[1], 1)])
        for k in range(chunks):
            yield ("hw_sync", named[k & 1])
            yield free(acc_free, k)
            yield full(bfull, k)
            yield ("work", t("mma") * 0.2)
            yield ("async", t("mma"), [(mma, 1)])
            if k + 1 < chunks:
                yield full(mma, k)
                yield ("async", t("load"), [(bfull, 1)])
                if k + 2 < chunks:
                    yield ("async", t("load"), [(xfull[k & 1], 1)])

    def state_warps():   # (eight warps that meet at hardware barriers of their own, in step)
        for k in range(chunks):
            yield ("work", t("state"))
            yield full(mma, k)
            yield ("work", t("state"))
            yield ("arrive", acc_free, 8)

    for i in range(3):
        sim.spawn(f"row{i}", row_warp())
    sim.spawn("issue", issuer())
    sim.spawn("state", state_warps())


ROLES = ("load", "rows", "mma", "state")


@pytest.mark.parametrize("chunks", [1, 2, 3, 4, 5, 8, 33])
def test_every_wait_is_sound_at_random_and_extreme_speeds(chunks):
    for seed in range(24):
        sim = StateSim(seed)
        speed = {r: 10.0 ** sim.rng.uniform(-2, 2) for r in ROLES}
        if seed < len(ROLES):
            speed = {r: 100.0 if r == ROLES[seed] else 0.01 for r in ROLES}
        build(sim, chunks, speed)
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
@pytest.mark.parametrize("chunks", [1, 2, 3, 5, 8])
def test_every_role_ends_when_arrivals_go_missing(chunks, rest):
    gave_up = 0
    for drop in range(1, 4 * chunks):
        for seed in range(4):
            sim = LossySim(seed, drop, rest)
            build(sim, chunks, SPEED)
            assert sim.run(), (drop, seed)
            gave_up += sim.gave_up
    assert gave_up > 0


def test_row_warps_that_go_on_would_not_let_them():
    # the row warps give up one wait per chunk, the issuing warp two: they overrun the barrier
    stuck = 0
    for drop in range(1, 20):
        sim = LossySim(drop, drop, rest=True)
        build(sim, 8, SPEED, broken=True)
        stuck += not sim.run()
    assert stuck > 0
