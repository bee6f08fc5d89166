"""The barrier protocol of the FP16-operand ChunkScan kernel (csrc/chunk_scan_f16.cu) on the host-side model of
test_scan_protocol_model.py: one CBq buffer and one xq buffer whose barriers come in pairs by the parity of the chunk, xq
rows expanded by the mask group behind its first tile.  Every wait is decided by parity alone and checked against the true
phase counts, and the two single buffers are watched: a load must not start while the tile before is still read.  `broken` names
variants that the model has to report."""
import pytest

from test_scan_protocol_model import Bar, Sim


def build(sim, ntiles, ntpu, speed, broken=None):
    rng = sim.rng
    B = lambda name, count, n: [Bar(f"{name}{i}", count) for i in range(n)]
    cb_full, cb_free, mq = B("CB_FULL", 1, 4), B("CB_FREE", 8, 4), B("MQ", 8, 4)
    tok_full, tok_free = B("TOK_FULL", 1, 4), B("TOK_FREE", 8, 4)
    acc, acc_free, afree = B("ACC", 1, 2), B("ACC_FREE", 8, 2), B("AFREE", 1, 2)
    ch_full, ch_free = B("CH_FULL", 1, 2), B("CH_FREE", 1, 2)
    x_raw, raw_free = B("X_RAW", 1, 2), Bar("RAW_FREE", 8)
    x_full, x_free = B("X_FULL", 8, 2), B("X_FREE", 8, 2)

    it_of = lambda n: n % ntpu
    unit = lambda n: n // ntpu
    cb_index = lambda n: (n & 3) if ntpu == 1 else ((0 if it_of(n) else 2) + ((n >> 1) & 1))
    t = lambda role: rng.expovariate(1.0) * speed[role]
    full = lambda bar, use: ("wait", bar, use & 1, use + 1)
    free = lambda bar, use: ("wait", bar, (use & 1) ^ 1, use)

    one = ntpu == 2 and ntiles == 2           # a CTA of one chunk: the mask groups take a tile each
    reading = [set() for _ in range(4)]       # the groups that read a slot of the scalar pack
    held = {}   # single buffer -> whose contents are being read

    def fill(name, who):
        assert held.get(name) is None, f"{name}: filled for {who} while {held[name]} is read"
        held[name] = who

    one_ch = broken == "one Cq/hq barrier pair"

    def prod_cb():
        for n in range(ntiles):
            ci = cb_index(n)
            if broken != "scalar pack without TOK_FREE":
                yield free(tok_free[n & 3], n >> 2)
            assert not reading[n & 3], f"TOK{n & 3}: filled for tile {n} while it is read"
            yield ("async", t("load"), [(tok_full[n & 3], 1)])
            if ntpu == 2 and it_of(n) == 0:
                if broken == "first CBq by its own pair":
                    yield free(cb_free[ci], n >> 2)
                elif n > 0:
                    yield full(cb_free[ci ^ 1], (n - 2) >> 2)
                fill("CB1", n)
            else:
                yield free(cb_free[ci], n >> 2)
            yield ("async", t("load"), [(cb_full[ci], 1)])
            yield ("work", t("producer"))

    def prod_ch():
        fill("XRAW", 0)
        yield ("async", t("load"), [(x_raw[0], 1)])
        for n in range(ntiles):
            if one_ch:
                yield free(ch_free[0], n)
            elif n > 0:
                yield full(ch_free[(n - 1) & 1], (n - 1) >> 1)
            yield ("async", t("load"), [(ch_full[0 if one_ch else n & 1], 1)])
            if it_of(n) == 0 and n + ntpu < ntiles:
                u = unit(n)
                if broken != "xq codes without RAW_FREE":
                    yield full(raw_free, u)
                fill("XRAW", u + 1)
                yield ("async", t("load"), [(x_raw[(u + 1) & 1], 1)])
            yield ("work", t("producer"))

    def issuer(par):
        for n in range(par, ntiles, 2):
            u = unit(n)
            yield free(acc_free[n & 1], n >> 1)
            yield full(ch_full[0], n) if one_ch else full(ch_full[par], n >> 1)
            yield ("work", t("mma"))
            yield ("async", t("mma"), [(ch_free[0 if one_ch else par], 1)])
            yield full(x_full[u & 1], u >> 1)
            yield full(mq[cb_index(n)], n >> 2)
            yield ("work", t("mma"))
            yield ("async", t("mma"), [(afree[n & 1], 1), (acc[n & 1], 1)])

    def mask(g):
        for n in range(ntiles):
            u = unit(n)
            if ((n if one else u) & 1) != g:
                continue
            yield full(tok_full[n & 3], n >> 2)
            reading[n & 3].add(g)
            yield full(cb_full[cb_index(n)], n >> 2)
            yield free(afree[n & 1], n >> 1)
            yield ("work", t("mask") * (1 + 2 * it_of(n)))
            reading[n & 3].discard(g)
            yield ("arrive", mq[cb_index(n)], 8)
            if ntpu == 2 and it_of(n) == 0:
                held["CB1"] = None
            yield ("arrive", cb_free[cb_index(n)], 8)
            if it_of(n) == 0:
                yield full(x_raw[u & 1], u >> 1)
                yield free(x_free[u & 1], u >> 1)
                yield ("work", t("mask"))
                held["XRAW"] = None
                yield ("arrive", x_full[u & 1], 8)
                yield ("arrive", raw_free, 8)

    def epilogue():
        for n in range(ntiles):
            u = unit(n)
            yield full(acc[n & 1], n >> 1)
            yield full(x_full[u & 1], u >> 1)
            yield full(tok_full[n & 3], n >> 2)
            reading[n & 3].add("epi")
            yield ("work", t("epilogue"))
            reading[n & 3].discard("epi")
            yield ("arrive", acc_free[n & 1], 8)
            yield ("arrive", tok_free[n & 3], 8)
            if it_of(n) + 1 == ntpu:
                yield ("arrive", x_free[u & 1], 8)

    for name, gen in [("prod_cb", prod_cb()), ("prod_ch", prod_ch()), ("mma0", issuer(0)), ("mma1", issuer(1)),
                      ("mask0", mask(0)), ("mask1", mask(1)), ("epi", epilogue())]:
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


@pytest.mark.parametrize("broken,where", [("first CBq by its own pair", "CB1"), ("one Cq/hq barrier pair", "CH_FULL"),
                                          ("xq codes without RAW_FREE", "XRAW"), ("scalar pack without TOK_FREE", "TOK")])
def test_broken_variants_are_reported(broken, where):
    """The first tiles' one CBq buffer guarded by the chunk before the last only; the odd tiles' MMA issuer on a barrier pair
    shared with the even ones', which polls the parity of phase 1 before phase 0 has completed; the xq codes of the next chunk
    requested without waiting for the mask group that expands the present ones; a slot of the scalar pack filled while a group
    reads it."""
    hit = 0
    for seed in range(24):
        sim = Sim(seed)
        speed = {r: 10.0 ** sim.rng.uniform(-2, 2) for r in ROLES}
        build(sim, 36, 2, speed, broken)
        try:
            sim.run()
        except AssertionError as e:
            assert where in str(e) or "deadlock" in str(e), e
            hit += 1
    assert hit > 0
