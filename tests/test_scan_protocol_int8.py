"""The barrier protocol of the int8 ChunkScan kernel (csrc/chunk_scan.cu) on the host-side model of
test_scan_protocol_model.py: two producers (one per tile of a chunk), one issuer per contraction, two mask groups, two
epilogue groups that hand xq back before they wait for the accumulators.  Every wait is decided by parity alone and checked
against the true phase counts: none is lapped, none passes early, every role finishes.  `broken` names variants that the model
has to report."""
import pytest

from test_scan_protocol_model import Bar, Sim


def build(sim, ntiles, ntpu, speed, broken=None):
    rng = sim.rng
    B = lambda name, count, n: [Bar(f"{name}{i}", count) for i in range(n)]
    cb_full, cb_free, mq = B("CB_FULL", 1, 4), B("CB_FREE", 1, 4), B("MQ", 8, 4)
    tok_full, tok_free = B("TOK_FULL", 1, 4), B("TOK_FREE", 8, 4)
    acc, acc_free = B("ACC", 2, 4), B("ACC_FREE", 4, 4)
    row_full, row_free = B("ROW_FULL", 9, 8), B("ROW_FREE", 4, 8)
    c_full, c_free = Bar("C_FULL", 1), Bar("C_FREE", 1)
    h_full, h_free = B("H_FULL", 1, 2), B("H_FREE", 1, 2)
    x_full, x_free = B("X_FULL", 1, 2), B("X_FREE", (4 if ntpu == 1 else 8) + (broken != "x_free without the MMAs"), 2)

    it_of = lambda n: n % ntpu
    unit = lambda n: n // ntpu
    cb_index = lambda n: (n & 3) if ntpu == 1 else ((0 if it_of(n) else 2) + ((n >> 1) & 1))
    t = lambda role: rng.expovariate(1.0) * speed[role]
    full = lambda bar, use: ("wait", bar, use & 1, use + 1)
    free = lambda bar, use: ("wait", bar, (use & 1) ^ 1, use)
    one = ntpu == 2 and ntiles == 2           # a CTA of one chunk: the mask groups take a tile each
    reading = [set() for _ in range(4)]       # the mask groups that read a slot of the scalar pack

    def producer(mine):
        for n0 in range(0, ntiles, ntpu):
            u = unit(n0)
            if mine == 0:
                if broken != "scalar pack without TOK_FREE":
                    yield free(tok_free[u & 3], u >> 2)
                assert not reading[u & 3], f"TOK{u & 3}: filled for chunk {u} while it is read"
                yield ("async", t("load"), [(tok_full[u & 3], 1)])
                yield free(h_free[u & 1], u >> 1)
                yield ("async", t("load"), [(h_full[u & 1], 1)])
            else:
                yield free(x_free[u & 1], u >> 1)
                yield ("async", t("load"), [(x_full[u & 1], 1)])
            if mine >= ntpu:
                continue
            n = n0 + mine
            yield free(cb_free[cb_index(n)], n >> 2)
            yield ("async", t("load"), [(cb_full[cb_index(n)], 1)])
            yield free(row_free[n & 7], n >> 3)
            yield ("async", t("load"), [(row_full[n & 7], 1)])
            yield ("work", t("producer"))

    def issuer_off():
        for n in range(ntiles):
            u = unit(n)
            yield free(c_free, n)
            yield ("async", t("load"), [(c_full, 1)])
            yield free(acc_free[n & 3], n >> 2)
            yield full(h_full[u & 1], u >> 1)
            yield full(c_full, n)
            yield ("work", t("mma"))
            done = [(c_free, 1), (acc[n & 3], 1)] + ([(h_free[u & 1], 1)] if it_of(n) + 1 == ntpu else [])
            yield ("async", t("mma"), done)

    def issuer_diag():
        for n in range(ntiles):
            u = unit(n)
            yield free(acc_free[n & 3], n >> 2)
            yield full(x_full[u & 1], u >> 1)
            yield full(mq[cb_index(n)], n >> 2)
            yield ("work", t("mma"))
            done = [(cb_free[cb_index(n)], 1), (acc[n & 3], 1)] + (
                [(x_free[u & 1], 1)] if it_of(n) + 1 == ntpu and broken != "x_free without the MMAs" else [])
            yield ("async", t("mma"), done)

    def mask(g):
        for n in range(ntiles):
            u = unit(n)
            if ((n if one else u) & 1) != g:
                continue
            yield full(tok_full[u & 3], u >> 2)
            reading[u & 3].add(g)
            yield full(cb_full[cb_index(n)], n >> 2)
            yield free(row_free[n & 7], n >> 3)
            yield ("work", t("mask") * (1 + 2 * it_of(n)))
            reading[u & 3].discard(g)
            yield ("arrive", mq[cb_index(n)], 8)
            yield ("arrive", row_full[n & 7], 8)
            if it_of(n) + 1 == ntpu:
                yield ("arrive", tok_free[u & 3], 8)

    def epilogue(eg):
        for n in range(eg, ntiles, 2):
            u = unit(n)
            yield full(x_full[u & 1], u >> 1)
            yield ("arrive", x_free[u & 1], 4)
            yield full(acc[n & 3], n >> 2)
            if broken == "epilogue waits on MQ":
                yield full(mq[cb_index(n)], n >> 2)
            yield full(row_full[n & 7], n >> 3)
            yield ("work", t("epilogue"))
            yield ("arrive", acc_free[n & 3], 4)
            yield ("arrive", row_free[n & 7], 4)

    for name, gen in [("prod0", producer(0)), ("prod1", producer(1)), ("off", issuer_off()), ("diag", issuer_diag()),
                      ("mask0", mask(0)), ("mask1", mask(1)), ("epi0", epilogue(0)), ("epi1", epilogue(1))]:
        sim.spawn(name, gen)


ROLES = ("load", "producer", "mma", "mask", "epilogue")


@pytest.mark.parametrize("ntpu", [1, 2])
@pytest.mark.parametrize("units", [1, 2, 3, 4, 5, 9, 35])
def test_every_wait_is_sound_at_random_and_extreme_speeds(ntpu, units):
    for seed in range(12):
        sim = Sim(seed)
        speed = {r: 10.0 ** sim.rng.uniform(-2, 2) for r in ROLES}
        if seed < len(ROLES):
            speed = {r: 100.0 if r == ROLES[seed] else 0.01 for r in ROLES}
        build(sim, units * ntpu, ntpu, speed)
        sim.run()


@pytest.mark.parametrize("broken,barrier,ntpu", [("epilogue waits on MQ", "MQ", 2), ("x_free without the MMAs", "X_F", 2),
                                                 ("scalar pack without TOK_FREE", "TOK", 1)])
def test_broken_variants_are_reported(broken, barrier, ntpu):
    """The mask barrier of a CBq buffer may complete for tile n + 4 while the epilogue group of tile n is busy with tile n - 2:
    nothing the epilogue releases stands between the two.  And an xq buffer that the epilogue alone hands back is filled again
    ahead of the MMAs that wait for its contents.  And a slot of the scalar pack is filled while the slower mask group reads it."""
    hit = 0
    for seed in range(24):
        sim = Sim(seed)
        speed = dict(load=0.1, producer=0.01, mma=0.01, mask=0.01, epilogue=5.0) if seed % 2 else \
            dict(load=0.1, producer=0.01, mma=5.0, mask=5.0, epilogue=0.01)
        build(sim, 36, ntpu, speed, broken)
        try:
            sim.run()
        except AssertionError as e:
            assert barrier in str(e) or "deadlock" in str(e)
            hit += 1
    assert hit > 0
