"""The variants that the launchers choose between and the exact fast paths inside the kernels, at the sizes and values
where they can go wrong, against the oracle.  Every comparison is bit for bit (the operation order of the library's
binary32 and binary64 arithmetic is part of its interface), so no tolerance is needed."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2608_21952_b200 import inputs
from paper_2608_21952_b200.inputs import SSDConfig

pytestmark = pytest.mark.gpu


def _ties(dt, A):
    # A = -1 and time steps on a grid of half binary32 units of the running sum: every prefix sum is exact in binary64
    # and about half of them lie exactly between two binary32 numbers
    A[:] = -1.0
    n = np.random.default_rng(5).integers(0, 5, dt.shape).astype(np.float64)
    dt[:] = (n * 2.0 ** -24).astype(np.float32)
    dt[:, 0] = 1.0


def _mixed(dt, A):
    dt[:, 1::3] *= -1.0


def _tiny(dt, A):
    dt *= np.float32(1e-36)


def _zero(dt, A):
    dt[:] = 0.0


def _huge(dt, A):
    dt[:, ::7] = np.float32(3e37)


@pytest.mark.parametrize("regime", [_ties, _mixed, _tiny, _zero, _huge], ids=lambda f: f.__name__[1:])
@pytest.mark.parametrize("H,Q", [(1, 64), (9, 128), (12, 256)])
def test_cumsum_scan_equals_the_sum_in_token_order(H, Q, regime):
    import gpu_harness as gh
    cfg = SSDConfig("cs", 2, 2 * Q, H, 64, 64, 1, Q, 0.02, 20.0, 31)
    q = orc.prepare_quantized(cfg, inputs.make_prefill(cfg))
    dt, A = q["dt"].reshape(2, 2 * Q, H).copy(), q["A"].copy()
    regime(dt[:, :Q], A)
    regime(dt[:, Q:], A)
    q["dt"], q["A"] = dt, A
    want = orc.chunk_cumsum(cfg, dt, A)
    _, _, taps = gh.gpu_fwd(cfg, q, taps=("cs",))
    assert np.array_equal(taps["cs"], want)


def test_cumsum_on_a_grid_that_fills_the_device():
    # 8 heads per block (the grid above takes 4), a last block with one head
    import gpu_harness as gh
    cfg = SSDConfig("cs_full", 2, 64 * 40, 17, 64, 64, 1, 64, 0.02, 20.0, 32)
    q = orc.prepare_quantized(cfg, inputs.make_prefill(cfg))
    want = orc.chunk_cumsum(cfg, q["dt"], q["A"])
    _, _, taps = gh.gpu_fwd(cfg, q, taps=("cs",))
    assert np.array_equal(taps["cs"], want)


@pytest.mark.parametrize("b,c,H,N,G,Q", [(1, 1, 1, 64, 1, 64), (2, 3, 9, 128, 1, 128), (1, 2, 16, 64, 2, 256), (3, 1, 150, 128, 1, 64)])
@pytest.mark.parametrize("with_init", [False, True])
def test_calibration_at_ragged_head_counts(b, c, H, N, G, Q, with_init):
    # 8 heads per block in the X_scaled pass (1 and 9 heads leave most of a block idle); whole heads and quarter heads per
    # CTA in the state pass
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("cal", b, c * Q, H, 64, N, G, Q, 0.02, 20.0, 33)
    t = inputs.make_prefill(cfg)
    init = inputs.make_init_state(cfg) * np.float32(3.0) if with_init else None
    q = orc.prepare_quantized(cfg, t, init)
    dims = bd.dims_of(cfg)
    dv = {k: gh.dev(q[k]) for k in ("xq", "Bq", "Cq", "s_x", "s_B", "s_C", "dt", "A")}
    s = [torch.full((n,), float("nan"), device="cuda") for n in (H * 64, G, H * 64)]
    bd.ssdi8_calibrate(dims, bd.make_fwd_args(init_state=gh.dev(init), **dv), *s, bd.alloc_workspace(dims))
    torch.cuda.synchronize()
    for got, name in zip(s, ("s_xs", "s_cb", "s_h")):
        assert np.array_equal(got.cpu().numpy(), np.asarray(q[name]).reshape(-1)), name


@pytest.mark.parametrize("R,Ch,I", [(1, 4, 1), (15, 516, 1), (16, 8, 64), (129, 2, 128)])
def test_quantiser_gives_all_zero_channels_a_step_of_one(R, Ch, I):
    import gpu_harness as gh
    v = np.random.default_rng(7).standard_normal((R, Ch, I)).astype(np.float32)
    v[:, ::2] = 0.0
    q, s = gh.gpu_quantize(v.reshape(R, Ch, I), R, Ch, I)
    qr, sr = orc.quantize(v.reshape(R, Ch, I), R, Ch, I, mode=1)
    assert np.array_equal(s, sr) and np.all(s[::2] == 1.0)
    assert np.array_equal(q.reshape(-1), np.asarray(qr).reshape(-1))


@pytest.mark.parametrize("R,Ch,I", [(1, 4, 1), (7, 36, 1), (9, 32, 1), (255, 1776, 1), (12800, 512, 1), (12801, 512, 1), (4100, 1028, 1), (300, 2400, 1),
                                    (1, 1, 64), (13, 3, 4), (5, 7, 12), (257, 37, 128), (258, 38, 128), (1023, 1, 128), (1025, 1, 128),
                                    (2047, 4, 128), (2049, 4, 128), (2048, 18, 64), (2048, 19, 64), (8, 2, 4096)])
def test_calibrating_quantiser_in_one_launch_and_in_three(R, Ch, I):
    # On either side of the lines of the dispatch; rows and columns that leave CTAs of a cluster, or threads, without any; the
    # largest value of a channel anywhere; a channel of zeros
    import gpu_harness as gh
    v = np.random.default_rng(R + Ch).standard_normal((R, Ch, I)).astype(np.float32)
    v[np.arange(Ch) * 7 % R, np.arange(Ch), np.arange(Ch) * 5 % I] = -(6.0 + np.arange(Ch, dtype=np.float32))
    v[:, Ch // 2] = 0.0
    q, s = gh.gpu_quantize(v, R, Ch, I)
    qr, sr = orc.quantize(v, R, Ch, I, mode=1)
    assert np.array_equal(s, sr)
    assert np.array_equal(q.reshape(-1), np.asarray(qr).reshape(-1))


@pytest.mark.parametrize("R,Ch,I", [(9, 32, 1), (4100, 1028, 1), (300, 2400, 1), (13, 3, 4), (257, 37, 128), (258, 38, 128), (2049, 4, 128)])
def test_a_channel_whose_quotient_is_zero_has_a_step_of_one(R, Ch, I):
    # One launch and three.  63 and 64 of the smallest number lie on either side of half of it times 127
    import gpu_harness as gh
    v = np.random.default_rng(R).standard_normal((R, Ch, I)).astype(np.float32)
    for ch, units in enumerate((63, 64, 7)):
        v[:, ch] = 0.0
        v[R // 2, ch, I // 2] = np.float32(-units * 2.0 ** -149)
    q, s = gh.gpu_quantize(v, R, Ch, I)
    qr, sr = orc.quantize(v, R, Ch, I, mode=1)
    assert np.array_equal(s, sr) and np.array_equal(q.reshape(-1), np.asarray(qr).reshape(-1))
    assert s[0] == 1.0 and s[1] == np.float32(2.0 ** -149) and s[2] == 1.0
    assert q[R // 2, 0, I // 2] == 0 and q[R // 2, 1, I // 2] == -64


@pytest.mark.parametrize("b,c,H,Q", [(1, 1, 1, 64), (2, 3, 9, 128), (1, 3, 17, 256)])
@pytest.mark.parametrize("regime", ["fast", "slow", "codes", "mixed"])
def test_calibration_skips_no_token_that_counts(b, c, H, Q, regime):
    # Which tokens can raise the largest |X_scaled| is decided by LUT_state: steep and nearly flat decay, codes that make a
    # channel's largest product sit on an early token, time steps of both signs and of zero
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("xs", b, c * Q, H, 64, 64, 1, Q, 0.02, 20.0, 61)
    t = inputs.make_prefill(cfg)
    t["A"] *= np.float32({"fast": 60.0, "slow": 0.001}.get(regime, 1.0))
    q = orc.prepare_quantized(cfg, t, None)
    if regime == "mixed":
        q["dt"] = q["dt"].copy()
        q["dt"].reshape(b, c * Q, H)[:, ::3] *= -1.0
        q["dt"].reshape(b, c * Q, H)[:, 1::5] = 0.0
    if regime == "codes":
        x = (np.abs(np.arange(b * c * Q * H * 64)) % 3).astype(np.int8).reshape(b, c * Q, H, 64)
        x[:, np.random.default_rng(1).integers(0, c * Q, 12)] = 127
        x[:, -1] = 0
        x[..., 5] = 0
        q["xq"] = x.reshape(np.asarray(q["xq"]).shape)
    want = orc.calibrate(cfg, q["xq"], q["Bq"], q["Cq"], q["s_x"], q["s_B"], q["s_C"], q["dt"], q["A"], None)
    dims = bd.dims_of(cfg)
    dv = {k: gh.dev(q[k]) for k in ("xq", "Bq", "Cq", "s_x", "s_B", "s_C", "dt", "A")}
    s = [torch.full((n,), float("nan"), device="cuda") for n in (H * 64, 1, H * 64)]
    bd.ssdi8_calibrate(dims, bd.make_fwd_args(**dv), *s, bd.alloc_workspace(dims))
    torch.cuda.synchronize()
    for got, ref in zip(s, want[:3]):
        assert np.array_equal(got.cpu().numpy(), np.asarray(ref).reshape(-1))


@pytest.mark.parametrize("b,c,H,Q", [(1, 11, 9, 256), (1, 12, 9, 256), (2, 5, 24, 128), (11, 1, 9, 256), (1, 10, 70, 256)])
@pytest.mark.parametrize("regime", ["slow", "codes"])
def test_calibration_skips_no_token_in_whole_chunks_and_in_parts(b, c, H, Q, regime):
    # Up to eleven chunks of few heads take 64 tokens to a block, more take the chunk
    test_calibration_skips_no_token_that_counts(b, c, H, Q, regime)


@pytest.mark.parametrize("R,Ch,I", [(9, 32, 1), (4100, 1028, 1), (300, 2400, 1), (13, 4, 4), (257, 37, 128), (258, 38, 128), (2049, 4, 128)])
def test_calibrating_quantiser_on_values_that_are_not_finite(R, Ch, I):
    # One launch and three: a NaN counts for nothing in a step size, an infinity makes it infinite (its own code is that of a NaN, all others
    # 0), a channel of NaNs has a step of 1.  Codes are those of the static mode under the same step sizes
    import gpu_harness as gh
    v = np.random.default_rng(R).standard_normal((R, Ch, I)).astype(np.float32)
    v[R // 2, 0, I // 2] = np.nan
    v[R - 1, 1, I - 1] = np.inf
    v[0, 2, 0], v[R - 1, 2, I - 1] = -np.inf, np.nan
    v[:, 3] = np.nan
    want = np.nanmax(np.abs(np.where(np.isnan(v), np.float32(0), v)), axis=(0, 2)) / np.float32(127)
    want[3] = 1.0
    q, s = gh.gpu_quantize(v, R, Ch, I)
    assert np.array_equal(s, want) and np.all(np.isinf(s[1:3])) and np.isfinite(s[0])
    assert np.array_equal(q, gh.gpu_quantize(v, R, Ch, I, scale=want, mode=0)[0])
    finite = np.isfinite(v[:, 1])
    assert not q.reshape(R, Ch, I)[:, 1][finite].any()


def test_calibration_passes_over_decays_and_step_sizes_that_are_not_finite():
    # LUT_state of a chunk with a NaN, an infinity of either sign or a very negative time step in it; step sizes of x that are infinite,
    # a NaN and zero
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("odd", 1, 5 * 256, 9, 64, 64, 1, 256, 0.02, 20.0, 74)
    q = orc.prepare_quantized(cfg, inputs.make_prefill(cfg), None)
    q["dt"], q["s_x"] = q["dt"].copy(), q["s_x"].copy()
    for k, bad in enumerate((np.nan, np.inf, -np.inf, -1e4)):
        q["dt"].reshape(1280, 9)[256 * k + 200, ::2] = bad
    q["s_x"][[5, 70, 71, 72]] = np.inf, np.nan, 0.0, np.inf
    want = orc.calibrate(cfg, q["xq"], q["Bq"], q["Cq"], q["s_x"], q["s_B"], q["s_C"], q["dt"], q["A"], None)
    dv = {k: gh.dev(q[k]) for k in ("xq", "Bq", "Cq", "s_x", "s_B", "s_C", "dt", "A")}
    s = [torch.full((n,), float("nan"), device="cuda") for n in (9 * 64, 1, 9 * 64)]
    bd.ssdi8_calibrate(bd.dims_of(cfg), bd.make_fwd_args(**dv), *s, bd.alloc_workspace(bd.dims_of(cfg)))
    torch.cuda.synchronize()
    for got, ref in zip(s[:2], want[:2]):
        assert np.array_equal(got.cpu().numpy(), np.asarray(ref).reshape(-1))


@pytest.mark.parametrize("step", [8e-41, 9.1e-41, 9.3e-41, 1e-39])
def test_calibration_skips_no_token_at_step_sizes_near_the_smallest(step):
    # 128 step sizes on either side of the normal range: the last token of the chunk has codes of 1, the one 64 before it codes of
    # 127 and a LUT_state of nearly the same size, every other token codes of 0
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("tiny", 1, 256, 8, 64, 64, 1, 256, 0.02, 20.0, 63)
    q = orc.prepare_quantized(cfg, inputs.make_prefill(cfg), None)
    x = np.zeros((256, 8, 64), np.int8)
    x[-1] = 1
    x[-65] = 127
    q.update(xq=x.reshape(np.asarray(q["xq"]).shape), s_x=np.full(512, step, np.float32), A=np.full(8, -1e-3, np.float32))
    q["dt"] = np.full_like(q["dt"], 0.5)
    want = orc.calibrate(cfg, q["xq"], q["Bq"], q["Cq"], q["s_x"], q["s_B"], q["s_C"], q["dt"], q["A"], None)
    dv = {k: gh.dev(q[k]) for k in ("xq", "Bq", "Cq", "s_x", "s_B", "s_C", "dt", "A")}
    s = [torch.full((n,), float("nan"), device="cuda") for n in (512, 1, 512)]
    bd.ssdi8_calibrate(bd.dims_of(cfg), bd.make_fwd_args(**dv), *s, bd.alloc_workspace(bd.dims_of(cfg)))
    torch.cuda.synchronize()
    assert np.all(np.asarray(want[0]) > 0) and np.all(np.asarray(want[0]) < 127 * step)
    for got, ref in zip(s, want[:3]):
        assert np.array_equal(got.cpu().numpy(), np.asarray(ref).reshape(-1))


@pytest.mark.parametrize("R,Ch", [(R, Ch) for R in (1, 3, 15, 17, 31, 33, 63, 2051) for Ch in (4, 508, 516)] + [(227, 113664), (227, 113668)])
def test_absmax_takes_every_row_into_account(R, Ch):
    # The largest value of each channel in a row of its own: remainders of the rows in flight, the row groups and the blocks
    import gpu_harness as gh
    v = np.random.default_rng(R).uniform(-1, 1, (R, Ch, 1)).astype(np.float32)
    v[np.arange(Ch) * 7 % R, np.arange(Ch), 0] = -(2.0 + np.arange(Ch, dtype=np.float32))
    q, s = gh.gpu_quantize(v, R, Ch, 1)
    qr, sr = orc.quantize(v, R, Ch, 1, mode=1)
    assert np.array_equal(s, sr)
    assert np.array_equal(q.reshape(-1), np.asarray(qr).reshape(-1))


@pytest.mark.parametrize("b,L,H,N,G,Q", [(1, 64, 1, 64, 1, 64), (1, 128, 7, 128, 1, 128), (2, 256, 8, 64, 2, 256), (1, 256, 17, 128, 1, 256),
                                         (2, 1024, 63, 64, 1, 128), (5, 1280, 21, 64, 3, 256), (4, 1024, 129, 64, 1, 64),
                                         (1, 192, 1, 64, 1, 64), (3, 256, 5, 128, 1, 64), (2, 384, 5, 128, 1, 128), (4, 1024, 33, 64, 3, 64),
                                         (2, 1024, 65, 128, 5, 128), (3, 1408, 50, 64, 2, 128)])
def test_layer_head_in_one_launch_and_in_two(b, L, H, N, G, Q):
    # On either side of the lines of the dispatch, head counts that leave a block of four heads partly idle: the layer call
    # gives the bits of the separate calls, whose ChunkCumsum and quantisers are launches of their own
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("lead", b, L, H, 64, N, G, Q, 0.02, 20.0, 48)
    t = inputs.make_prefill(cfg)
    T, HP = b * L, H * 64
    s = {"s_x": np.full(HP, 0.05), "s_B": np.full(G, 0.03), "s_C": np.full(G, 0.03), "s_xs": np.full(HP, 0.002),
         "s_cb": np.full(G, 0.4), "s_h": np.full(HP, 0.02)}
    s = {k: gh.dev(v.astype(np.float32)) for k, v in s.items()}
    dv = {k: gh.dev(np.asarray(v, np.float32)) for k, v in t.items()}
    codes = {k: torch.empty(n, dtype=torch.int8, device="cuda") for k, n in (("xq", (T, HP)), ("Bq", (T, G * N)), ("Cq", (T, G * N)))}
    bd.ssdi8_quantize_act(dv["x"], T, HP, 1, s["s_x"], 0, codes["xq"])
    bd.ssdi8_quantize_act(dv["B"], T, G, N, s["s_B"], 0, codes["Bq"])
    bd.ssdi8_quantize_act(dv["C"], T, G, N, s["s_C"], 0, codes["Cq"])
    dims = bd.dims_of(cfg)
    out = []
    for layer in (False, True):
        y = torch.full((b, L, H, 64), float("nan"), device="cuda")
        fin = torch.full((b, H, 64, N), float("nan"), device="cuda")
        status = torch.full((1,), 5, dtype=torch.int32, device="cuda")
        rest = dict(dt=dv["dt"], A=dv["A"], D=dv["D"], y=y, final_state=fin, status=status, **s)
        if layer:
            ws = torch.empty(bd.ssdi8_layer_fwd_workspace_bytes(dims), dtype=torch.uint8, device="cuda")
            bd.ssdi8_layer_fwd(dims, bd.make_layer_args(x=dv["x"], B=dv["B"], C=dv["C"], **rest), ws)
        else:
            bd.ssdi8_chunk_scan_fwd(dims, bd.make_fwd_args(**codes, **rest), bd.alloc_workspace(dims))
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        out.append((y, fin))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("b,L,H,Q,head", [(1, 128, 4, 64, 2), (1, 192, 4, 64, 1), (1, 1024, 4, 64, 1), (1, 1088, 4, 64, 2), (2, 1024, 63, 64, 2),
                                          (2, 1024, 64, 64, 1), (4, 1024, 128, 64, 1), (4, 1024, 129, 64, 2), (8, 256, 1, 128, 2), (1, 384, 8, 128, 1),
                                          (1, 1152, 4, 128, 2), (2, 1024, 64, 128, 1), (4, 1024, 129, 128, 2), (1, 1024, 4, 256, 2),
                                          (2, 1024, 63, 256, 2), (2, 1024, 64, 256, 1), (4, 1024, 128, 256, 1), (4, 1024, 129, 256, 2)])
def test_launches_of_the_layer_head(b, L, H, Q, head):
    # ChunkCumsum and the quantisers are one launch for three or more chunks of up to 128 with at most 4096 tokens x heads, and for
    # 128 to 512 thousand: a layer call then has as many kernels as Algorithm 2 alone, elsewhere one more
    import torch
    rt = pytest.importorskip("cuda.bindings.runtime")
    from paper_2608_21952_b200 import binding as bd
    T, HP = b * L, H * 64
    dims = bd.Dims(b, L, H, 64, 64, 1, Q)
    new = lambda *n: torch.ones(*n, device="cuda")  # noqa: E731
    s = {"s_x": new(HP), "s_B": new(1), "s_C": new(1), "s_xs": new(HP), "s_cb": new(1), "s_h": new(HP)}
    rest = dict(dt=new(T, H), A=-new(H), D=new(H), y=new(b, L, H, 64), final_state=new(b, H, 64, 64), **s)
    codes = {k: torch.ones(n, dtype=torch.int8, device="cuda") for k, n in (("xq", (T, HP)), ("Bq", (T, 64)), ("Cq", (T, 64)))}
    fwd, layer = bd.make_fwd_args(**codes, **rest), bd.make_layer_args(x=new(T, HP), B=new(T, 64), C=new(T, 64), **rest)
    ws = bd.alloc_workspace(dims)
    layer_ws = torch.empty(bd.ssdi8_layer_fwd_workspace_bytes(dims), dtype=torch.uint8, device="cuda")

    def kernels(call):
        g = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(g):
            call()
        err, _, n = rt.cudaGraphGetNodes(g.raw_cuda_graph())
        assert int(err) == 0
        return n

    alone = kernels(lambda: bd.ssdi8_chunk_scan_fwd(dims, fwd, ws))
    assert kernels(lambda: bd.ssdi8_layer_fwd(dims, layer, layer_ws)) == alone + head - 1


@pytest.mark.parametrize("Q,N,H", [(256, 128, 5), (256, 64, 148), (256, 128, 149), (128, 128, 3)])
def test_scan_with_one_chunk_per_cta(Q, N, H):
    # As many chunks as SMs, one more, and few: with two tiles per chunk the mask groups take one each where a CTA has one chunk (with
    # chunks of 128, a tile each as it is, one group has all the work)
    import gpu_harness as gh
    cfg = SSDConfig("one", 1, Q, H, 64, N, 1, Q, 0.02, 20.0, 47)
    q = orc.prepare_quantized(cfg, inputs.make_prefill(cfg))
    y, fin, taps = gh.gpu_fwd(cfg, q, taps=("Mq", "acc_diag"))
    _, fin_ref, ref = orc.ssdi8_fwd(cfg, q["xq"], q["Bq"], q["Cq"], q["s_x"], q["s_B"], q["s_C"], q["dt"], q["A"], q["D"], None,
                                    q["s_xs"], q["s_cb"], q["s_h"], taps=("Mq", "acc_diag"))
    assert np.array_equal(fin, fin_ref)
    for name in taps:
        assert np.array_equal(taps[name], ref[name]), name
    assert np.array_equal(y, gh.gpu_fwd(cfg, q, taps=())[0])


@pytest.mark.parametrize("b,c,H,G", [(9, 1, 80, 1), (5, 2, 129, 1), (2, 7, 130, 2), (6, 3, 40, 8), (1, 9, 256, 1), (14, 1, 8, 1)],
                         ids=lambda v: str(v))
@pytest.mark.parametrize("flags", [0, 2 | 4], ids=["default", "int8_state_y_fp16"])
def test_host_pipeline_cuts_equal_the_device_call(b, c, H, G, flags):
    # several whole elements per slice with a ragged last one, one element per slice, elements in two, three and more
    # slices (a short last one among them), B, C and dt in one piece per element and in several: bit for bit
    import torch
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("host_cut", b, c * 128, H, 64, 64, G, 128, 0.02, 20.0, 34)
    dims = bd.dims_of(cfg)
    g = torch.Generator().manual_seed(3)
    T, HP = cfg.tokens, cfg.channels
    r = lambda *s: torch.randn(*s, generator=g)
    host = {"x": r(T, HP), "B": r(T, G * 64), "C": r(T, G * 64), "dt": torch.nn.functional.softplus(r(T, H) - 3.0)}
    host = {k: v.pin_memory() for k, v in host.items()}
    dv = {k: v.cuda() for k, v in host.items()}
    init = r(b, H, 64, 64).cuda()
    par = {"A": -torch.exp(r(H)).cuda(), "D": r(H).cuda(), "s_x": torch.full((HP,), 0.03), "s_B": torch.full((G,), 0.03),
           "s_C": torch.full((G,), 0.03), "s_xs": torch.full((HP,), 0.002), "s_cb": torch.full((G,), 0.4),
           "s_h": torch.full((HP,), 0.02)}
    par = {k: v.cuda() for k, v in par.items()}
    ydt = torch.float16 if flags & 4 else torch.float32
    y_d, fin_d = torch.empty(T, HP, dtype=ydt, device="cuda"), torch.empty_like(init)
    lws = torch.empty(bd.ssdi8_layer_fwd_workspace_bytes(dims, flags), dtype=torch.uint8, device="cuda")
    bd.ssdi8_layer_fwd(dims, bd.make_layer_args(y=y_d, final_state=fin_d, init_state=init, **dv, **par), lws, flags=flags)
    scratch = torch.empty(bd.ssdi8_layer_fwd_host_scratch_bytes(dims, flags), dtype=torch.uint8, device="cuda")
    for with_state in (True, False, True):
        y_h = torch.full((T, HP), float("nan"), dtype=ydt).pin_memory()
        fin_h = torch.full(init.shape, float("nan")).pin_memory()
        st = torch.full((1,), -99, dtype=torch.int32).pin_memory()
        bd.ssdi8_layer_fwd_host(dims, bd.make_host_args(y=y_h, final_state=fin_h if with_state else None, status=st,
                                                        init_state=init, **host, **par), scratch, flags=flags)
        torch.cuda.synchronize()
        assert int(st[0]) == 0
        assert torch.equal(y_h, y_d.cpu())
        assert not with_state or torch.equal(fin_h, fin_d.cpu())


@pytest.mark.parametrize("cfg", [SSDConfig("split_small", 1, 8 * 64, 1, 64, 128, 1, 64, 0.02, 20.0, 35),
                                 SSDConfig("split_deep", 2, 17 * 64, 3, 64, 64, 1, 64, 0.02, 20.0, 36),
                                 SSDConfig("split_q256", 1, 9 * 256, 5, 64, 128, 1, 256, 0.02, 20.0, 37),
                                 SSDConfig("split_edge", 1, 12 * 64, 49, 64, 64, 7, 64, 0.02, 20.0, 38),
                                 SSDConfig("fused_edge", 2, 12 * 64, 25, 64, 64, 5, 64, 0.02, 20.0, 39),
                                 SSDConfig("fused_eight", 2, 8 * 64, 19, 64, 128, 1, 64, 0.02, 20.0, 41),
                                 SSDConfig("fused_short", 1, 3 * 128, 2, 64, 128, 1, 128, 0.02, 20.0, 40),
                                 SSDConfig("fused_one", 2, 256, 30, 64, 128, 2, 256, 0.02, 20.0, 42),
                                 SSDConfig("fused_q256", 1, 4 * 256, 60, 64, 64, 1, 256, 0.02, 20.0, 43),
                                 SSDConfig("quarters_last", 2, 4 * 64, 50, 64, 64, 1, 64, 0.02, 20.0, 44),
                                 SSDConfig("whole_first", 1, 4 * 64, 101, 64, 64, 1, 64, 0.02, 20.0, 45)], ids=lambda c: c.name)
@pytest.mark.parametrize("fast", [False, True])
def test_state_kernels_on_both_sides_of_the_dispatch(cfg, fast):
    # With 12 chunks 49 (batch, head) pairs are the last that take ChunkState + StatePassing on 148 SMs, 50 the first that do
    # not; with 8 chunks 37 and 38; 17 and 9 chunks leave one after two and one batches of eight.  The fused kernel shares
    # the live rows of a chunk among its warps: heads of different decay have any number of live slabs, and with very
    # fast decay whole slabs and whole chunks re-quantise to zero
    from test_gpu_parity import check_fwd

    def decay(t):
        t["A"] *= np.float32(60.0)

    check_fwd(cfg, init=inputs.make_init_state(cfg, 0.5), mutate=decay if fast else None)


@pytest.mark.parametrize("cfg", [SSDConfig("whole_few", 2, 3 * 128, 50, 64, 128, 2, 128, 0.02, 20.0, 51),
                                 SSDConfig("whole_alone", 1, 2 * 64, 101, 64, 128, 1, 64, 0.02, 20.0, 52),
                                 SSDConfig("slices_64", 1, 3 * 256, 9, 64, 128, 3, 256, 0.02, 20.0, 53),
                                 SSDConfig("slices_32", 1, 13 * 64, 5, 64, 128, 1, 64, 0.02, 20.0, 54),
                                 SSDConfig("slices_n64", 1, 5 * 128, 7, 64, 64, 1, 128, 0.02, 20.0, 55),
                                 SSDConfig("many", 3, 2 * 256, 100, 64, 64, 2, 256, 0.02, 20.0, 56),
                                 SSDConfig("slices_last", 5, 2 * 64, 90, 64, 128, 1, 64, 0.02, 20.0, 57),
                                 SSDConfig("cluster", 1, 8 * 64, 1, 64, 64, 1, 64, 0.02, 20.0, 58),
                                 SSDConfig("cluster_q256", 2, 8 * 256, 3, 64, 128, 3, 256, 0.02, 20.0, 59),
                                 SSDConfig("cluster_most", 1, 8 * 128, 37, 64, 128, 1, 128, 0.02, 20.0, 60),
                                 SSDConfig("cluster_beyond", 1, 8 * 64, 38, 64, 64, 2, 64, 0.02, 20.0, 62)], ids=lambda c: c.name)
@pytest.mark.parametrize("decay", [0.002, 1.0, 60.0])
def test_fused_state_kernel_with_few_and_many_sequences(cfg, decay):
    # Up to two CTAs per SM (whole heads, slices of 32 and of 64 state columns), three, and a last wave in slices; decay rates
    # at which every slab of every chunk is live, some are, and none is; eight chunks, whose binary32 states take a cluster per
    # sequence where there are few.  INT8 states always take this kernel, and the codes of
    # the states that enter the chunks and the final state are all that it writes (the taps' instance is another kernel).
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    t = inputs.make_prefill(cfg)
    t["A"] *= np.float32(decay)
    init = inputs.make_init_state(cfg, 0.5)
    q = orc.prepare_quantized(cfg, t, init)
    for gpu_flags, flags in ((0, 0), (bd.FLAG_INT8_STATE, orc.FLAG_INT8_STATE)):
        _, fin_ref, ref = orc.ssdi8_fwd(cfg, q["xq"], q["Bq"], q["Cq"], q["s_x"], q["s_B"], q["s_C"], q["dt"], q["A"], q["D"], None,
                                        q["s_xs"], q["s_cb"], q["s_h"], init, taps=("hq",), flags=flags)
        _, fin, got = gh.gpu_fwd(cfg, q, taps=("hq",), flags=gpu_flags)
        assert np.array_equal(got["hq"], ref["hq"])
        assert np.array_equal(fin, fin_ref)


@pytest.mark.parametrize("cfg", [SSDConfig("six_slabs", 1, 6 * 64, 7, 64, 64, 1, 64, 0.02, 20.0, 65),
                                 SSDConfig("seven_slabs", 1, 7 * 64, 7, 64, 64, 1, 64, 0.02, 20.0, 66),
                                 SSDConfig("three_of_two", 1, 3 * 128, 37, 64, 128, 1, 128, 0.02, 20.0, 67),
                                 SSDConfig("four_of_two", 1, 4 * 128, 5, 64, 128, 1, 128, 0.02, 20.0, 68),
                                 SSDConfig("two_of_four", 1, 2 * 256, 59, 64, 128, 1, 256, 0.02, 20.0, 69),
                                 SSDConfig("whole_after", 1, 3 * 64, 60, 64, 128, 2, 64, 0.02, 20.0, 70),
                                 SSDConfig("nearly_all_sms", 1, 2 * 128, 119, 64, 128, 1, 128, 0.02, 20.0, 71),
                                 SSDConfig("nearly_two_each", 2, 256, 134, 64, 128, 1, 256, 0.02, 20.0, 72),
                                 SSDConfig("two_each", 2, 256, 133, 64, 64, 1, 256, 0.02, 20.0, 73)], ids=lambda c: c.name)
@pytest.mark.parametrize("decay", [0.002, 60.0])
def test_fused_state_kernel_on_short_calls(cfg, decay):
    # Calls whose slabs the ring of six holds at once and calls with a slab more; slices and whole heads of two and three chunks; one
    # chunk of 256 on either side of 1.8 CTAs per SM.  Every slab live, and none
    test_fused_state_kernel_with_few_and_many_sequences(cfg, decay)


@pytest.mark.parametrize("b,H", [(5, 89), (5, 99)])
@pytest.mark.parametrize("decay", [0.002, 1.0, 60.0])
def test_a_last_wave_of_n_64_in_slices(b, H, decay):
    # 1 and 51 sequences beyond three per SM: state columns in slices of 32 beside whole heads, binary32 and INT8 states and the
    # calibration of the same shape
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("slices_last_n64", b, 2 * 64, H, 64, 64, 1, 64, 0.02, 20.0, 76)
    test_fused_state_kernel_with_few_and_many_sequences(cfg, decay)
    t = inputs.make_prefill(cfg)
    t["A"] *= np.float32(decay)
    init = inputs.make_init_state(cfg, 0.5)
    q = orc.prepare_quantized(cfg, t, init)
    dv = {k: gh.dev(q[k]) for k in ("xq", "Bq", "Cq", "s_x", "s_B", "s_C", "dt", "A")}
    s = [torch.full((n,), float("nan"), device="cuda") for n in (H * 64, 1, H * 64)]
    bd.ssdi8_calibrate(bd.dims_of(cfg), bd.make_fwd_args(init_state=gh.dev(init), **dv), *s, bd.alloc_workspace(bd.dims_of(cfg)))
    torch.cuda.synchronize()
    for got, name in zip(s, ("s_xs", "s_cb", "s_h")):
        assert np.array_equal(got.cpu().numpy(), np.asarray(q[name]).reshape(-1)), name


def test_the_tap_of_x_scaled_reaches_the_last_of_many_chunks():
    # Q(X_scaled) of a chunk depends on nothing outside it: the same chunk 32 770 times over has the same codes 32 770 times (more
    # chunks than 16 bits of a signed index count).  INT8 states, which take the chunk-sequential kernel at any length.
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    c = 32770
    one = SSDConfig("one", 1, 64, 1, 64, 64, 1, 64, 0.02, 20.0, 64)
    q = orc.prepare_quantized(one, inputs.make_prefill(one))
    want = gh.dev(orc.ssdi8_fwd(one, q["xq"], q["Bq"], q["Cq"], q["s_x"], q["s_B"], q["s_C"], q["dt"], q["A"], q["D"], None, q["s_xs"],
                                q["s_cb"], q["s_h"], None, taps=("Xsq",), flags=orc.FLAG_INT8_STATE)[2]["Xsq"]).reshape(64, 64)
    dims = bd.Dims(1, 64 * c, 1, 64, 64, 1, 64)
    dv = {k: gh.dev(q[k]) for k in ("s_x", "s_B", "s_C", "A", "s_xs", "s_cb", "s_h")}
    dv.update({k: gh.dev(q[k]).reshape(64, -1).repeat(c, 1) for k in ("xq", "Bq", "Cq", "dt")})
    tap = torch.full((c, 64, 64), 99, dtype=torch.int8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    phases = bd.PHASE_CUMSUM | bd.PHASE_CHUNK_STATE | bd.PHASE_STATE_PASSING
    bd.ssdi8_chunk_scan_fwd(dims, bd.make_fwd_args(y=torch.empty(4, device="cuda"), tap_Xsq=tap, status=status, **dv),
                            bd.alloc_workspace(dims, flags=bd.FLAG_INT8_STATE), flags=bd.FLAG_INT8_STATE | phases)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert torch.equal(tap, want.expand(c, 64, 64))


def _near_ties():
    # Pairs (v, alpha) whose quotient lies within 8 / alpha's significand of the midpoint between k + 1/2 and a neighbour
    # in binary32: where a quotient formed from a reciprocal could fall on the other side.
    v, a = [], []
    for k in range(128):
        h = np.float32(k + 0.5)
        for nb in (np.nextafter(h, np.float32(np.inf)), np.nextafter(h, np.float32(0))):
            mid = (float(h) + float(nb)) / 2
            M = int(np.ldexp(np.frexp(mid)[0], 25))
            for s in (24, 25):
                for j in range(-8, 9):
                    A = j * pow(M, -1, 1 << s) % (1 << s)
                    V = (M * A - j) >> s
                    if 1 << 23 <= A < 1 << 24 and 1 << 23 <= V < 1 << 24:
                        a.append(A)
                        v.append(np.ldexp(V, int(np.rint(np.log2(mid * A / V)))))
    return np.float32(v), np.float32(a)


@pytest.mark.parametrize("dtype", ["float32", "float16", "bfloat16", "near ties"])
def test_entry_quantiser_codes_are_those_of_the_division(dtype):
    # Every finite 16-bit pattern (and the same values as binary32, with their neighbours) under step sizes where quotients
    # are ties, near-ties, saturated, overflowing or underflowing, and under step sizes that take the divisions.  The
    # reference is the definition, rne(fdiv(v, alpha)) saturated: numpy's binary32 division is correctly rounded.
    import torch
    from paper_2608_21952_b200 import binding as bd
    pat = np.arange(65536, dtype=np.uint16)
    if dtype == "bfloat16":
        vals = (pat.astype(np.uint32) << 16).view(np.float32)
    else:
        vals = pat.view(np.float16).astype(np.float32)
    vals = vals[np.isfinite(vals)]
    if dtype == "float32":
        vals = np.concatenate([vals, np.nextafter(vals, np.float32(np.inf)), np.nextafter(vals, np.float32(-np.inf))])
    vals = vals[np.isfinite(vals)]
    rng = np.random.default_rng(9)
    alpha = np.concatenate([np.float32([1.0, 0.5, 2.0 ** -5, 3.0, 1.0 / 127, 1.0 / 3, 0.1, 1e-30, 9e-31, 1e30, 1.1e30, 1e-38, 1e-42,
                                        1e-20, 5e4, 2.0 ** -9 / 127]),
                            np.abs(rng.choice(vals[vals != 0], 32)).astype(np.float32) / np.float32(127),
                            np.exp(rng.uniform(-9, 3, 80)).astype(np.float32)]).astype(np.float32)
    if dtype == "near ties":
        dtype, (vals, alpha) = "float32", _near_ties()
        n = alpha.size // 16 * 16
        vals, alpha = vals[:n], alpha[:n]
    D, T = alpha.size, (vals.size + 7) // 8 * 8 + 3          # a ragged last round
    col = np.resize(vals, T)
    x = np.repeat(col[:, None], D, axis=1)
    t = torch.from_numpy(np.concatenate([x, np.zeros((T, 32), np.float32)], axis=1)).to(getattr(torch, dtype)).cuda()
    s_x = torch.from_numpy(alpha).cuda()
    one = torch.ones(1, device="cuda")
    out = [torch.empty(T, w, dtype=torch.int8, device="cuda") for w in (D, 16, 16)]
    bd.ssdi8_quantize_entry(t, T, D, 1, 16, s_x, one, one, *out)
    with np.errstate(all="ignore"):
        want = np.clip(np.rint(x / alpha), -127, 127).astype(np.int8)
    got = out[0].cpu().numpy()
    bad = np.argwhere(got != want)
    assert bad.size == 0, (len(bad), col[bad[0][0]], alpha[bad[0][1]], got[tuple(bad[0])], want[tuple(bad[0])])


def _random_codes(cfg, seed):
    # int8 tensors and step sizes for chunk_scan_fwd without the oracle's calibration
    rng = np.random.default_rng(seed)
    T, H, G, N = cfg.tokens, cfg.nheads, cfg.ngroups, cfg.dstate
    r = lambda *s: rng.integers(-127, 128, s).astype(np.int8)
    c = lambda n, v: np.full(n, v, np.float32)
    return dict(xq=r(T, H * 64), Bq=r(T, G * N), Cq=r(T, G * N), s_x=c(H * 64, 0.03), s_B=c(G, 0.03), s_C=c(G, 0.03),
                s_xs=c(H * 64, 0.002), s_cb=c(G, 0.4), s_h=c(H * 64, 0.02), D=rng.standard_normal(H).astype(np.float32),
                dt=np.log1p(np.exp(rng.standard_normal((T, H)) - 3.0)).astype(np.float32),
                A=-np.exp(rng.uniform(0.0, 2.7, H)).astype(np.float32),
                init=rng.standard_normal((cfg.batch, H, 64, N)).astype(np.float32))


@pytest.mark.parametrize("Q", [64, 128, 256])
@pytest.mark.parametrize("taps", [("acc_off", "acc_diag"), ("Mq", "rowmax")], ids="+".join)
def test_output_does_not_depend_on_the_pace_of_the_epilogue(Q, taps):
    # Several chunks per CTA, with the epilogue (or the mask) held up by the stores of taps: the same bits as without
    import gpu_harness as gh
    cfg = SSDConfig("pace", 2, 6 * 256, 101, 64, 64, 1, Q, 0.02, 20.0, 46)
    q = _random_codes(cfg, 46)
    want = gh.gpu_fwd(cfg, q, taps=())[:2]
    for _ in range(3):
        y, fin, _ = gh.gpu_fwd(cfg, q, taps=taps)
        assert np.array_equal(y, want[0]) and np.array_equal(fin, want[1])


@pytest.mark.parametrize("flag", ["INT8", "FP16"])
@pytest.mark.parametrize("Q", [128, 256])
def test_few_heads_give_the_bits_of_the_same_heads_among_many(Q, flag):
    # One chunk per CTA against several; with chunks of 256 its mask groups take a tile each there, with chunks of 128 (one tile) the
    # first group has it
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    flags = bd.FLAG_FP16_OPERAND if flag == "FP16" else 0
    many = SSDConfig("many", 1, Q, 320, 64, 128, 1, Q, 0.02, 20.0, 49)
    q = _random_codes(many, 49)
    want = gh.gpu_fwd(many, q, taps=(), flags=flags)[:2]
    few = SSDConfig("few", 1, Q, 7, 64, 128, 1, Q, 0.02, 20.0, 49)
    cut = dict(q)
    for k in ("xq", "dt", "A", "D", "s_x", "s_xs", "s_h", "init"):
        v = np.asarray(q[k])
        axis = [n for n, size in enumerate(v.shape) if size in (320, 320 * 64)][0]
        cut[k] = np.ascontiguousarray(np.take(v, np.arange(v.shape[axis] // 320 * 7), axis=axis))
    y, fin, _ = gh.gpu_fwd(few, cut, taps=(), flags=flags)
    assert np.array_equal(y, want[0][:, :, :7]) and np.array_equal(fin, want[1][:, :7])


@pytest.mark.parametrize("softplus", [False, True])
@pytest.mark.parametrize("Q", [64, 128, 256])
def test_cumsum_of_a_chunk_does_not_depend_on_the_number_of_chunks(Q, softplus):
    # Blocks of four heads for up to half of the SMs (74 blocks of a B200: 37 chunks of 5 heads), for more of them, and blocks of
    # eight: cs and y of the first chunks are the same
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("long", 1, 149 * Q, 5, 64, 64, 1, Q, 0.02, 20.0, 50)
    q = _random_codes(cfg, 50)
    bias = np.linspace(-4, -2, 5).astype(np.float32) if softplus else None
    flags = bd.FLAG_DT_SOFTPLUS if softplus else 0
    runs = []
    for c in (37, 38, 149):
        short = SSDConfig("short", 1, c * Q, 5, 64, 64, 1, Q, 0.02, 20.0, 50)
        cut = {k: np.ascontiguousarray(v[:c * Q]) if k in ("xq", "Bq", "Cq", "dt") else v for k, v in q.items()}
        y, _, taps = gh.gpu_fwd(short, cut, taps=("cs",), flags=flags, dt_bias=bias)
        runs.append((y[:, :37 * Q], taps["cs"][:, :, :37]))
    for y, cs in runs[1:]:
        assert np.array_equal(y, runs[0][0]) and np.array_equal(cs, runs[0][1])
    if not softplus:
        ref = np.cumsum((q["dt"][:37 * Q].astype(np.float64) * q["A"].astype(np.float64)).reshape(37, Q, 5), axis=1).astype(np.float32)
        assert np.array_equal(runs[0][1][0], ref.transpose(2, 0, 1))


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("Q", [64, 128, 256])
@pytest.mark.parametrize("flag", ["INT8", "FP16"])
def test_a_time_step_that_is_not_finite_does_not_reach_earlier_tokens(Q, value, flag):
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    flags = bd.FLAG_FP16_OPERAND if flag == "FP16" else 0
    cfg = SSDConfig("causal", 1, 2 * Q, 3, 64, 64, 1, Q, 0.02, 20.0, 47)
    q = _random_codes(cfg, 47)
    want = gh.gpu_fwd(cfg, q, taps=(), flags=flags)[0]
    for j in (0, 5, 15, Q - 1, Q + 8, 2 * Q - 10):
        dt = q["dt"].copy()
        dt[j, 1] = value
        y = gh.gpu_fwd(cfg, dict(q, dt=dt), taps=(), flags=flags)[0]
        assert np.array_equal(y[:, :j], want[:, :j]), j
        assert np.array_equal(y[:, :, ::2], want[:, :, ::2])


@pytest.mark.parametrize("dtype", ["float32", "float16", "bfloat16"])
def test_codes_do_not_depend_on_the_row(dtype):
    # The same values in every row, in full rounds of eight rows and in the remainder: NaNs of both signs, infinities,
    # values beyond the range of the quotient among them
    import torch
    from paper_2608_21952_b200 import binding as bd
    v = np.array([0x7fc00000, 0xffc00000, 0x7f800000, 0xff800000, 0x7f7fffff, 0xff7fffff, 0, 0x80000000], np.uint32).view(np.float32)
    D, T = 64, 8 + 7
    row = np.concatenate([np.resize(v, D), np.zeros(32, np.float32)])
    bits = row.view(np.int32)
    t = torch.from_numpy(np.tile(bits, (T, 1))).cuda().view(torch.float32)
    if dtype == "bfloat16":    # (torch's conversion drops the sign of a NaN)
        t = torch.from_numpy(np.tile((bits >> 16).astype(np.int16), (T, 1))).cuda().view(torch.bfloat16)
    elif dtype == "float16":
        t = t.half()
        t[:, 1::8].view(torch.int16).fill_(-512)   # 0xfe00: a negative NaN
    one = torch.ones(1, device="cuda")
    out = [torch.empty(T, w, dtype=torch.int8, device="cuda") for w in (D, 16, 16)]
    s_x = torch.from_numpy(np.repeat(np.float32([0.03, 1.0, 1e-42, 3e-30, 7e29, np.inf, 0.5, 127.0]), 8)).cuda()
    bd.ssdi8_quantize_entry(t.contiguous(), T, D, 1, 16, s_x, one, one, *out)
    got = out[0].cpu().numpy()
    assert np.array_equal(got, np.tile(got[8:9], (T, 1)))
    assert np.all(got[:, 0::8] == 127) and np.all(got[:, 1::8] == 127)   # a NaN of either sign, as by division
    if dtype == "float32":
        q = torch.empty(T, D, dtype=torch.int8, device="cuda")
        bd.ssdi8_quantize_act(t[:, :D].contiguous(), T, D, 1, s_x, 0, q)
        assert np.array_equal(q.cpu().numpy(), got)


@pytest.mark.parametrize("chunks", [1, 3, 4, 5, 7, 8, 15, 16, 17, 24, 25, 31, 32, 33, 40])
@pytest.mark.parametrize("prev", [None, "own", "loc", "before loc"])
def test_state_passing_batches(chunks, prev):
    # every remainder of the batches of four and eight chunks and of the batch ahead; prev absent, of its own, over loc, and
    # starting one chunk before loc
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("batches", 1, 64 * chunks, 3, 64, 64, 1, 64, 0.02, 20.0, 48)
    rng = np.random.default_rng(chunks)
    per = 3 * 64 * 64
    loc = rng.standard_normal((1, chunks, 3, 64, 64)).astype(np.float32)
    gamma = rng.uniform(0, 1, (1, 3, chunks)).astype(np.float32)
    init = rng.standard_normal((1, 3, 64, 64)).astype(np.float32)
    s_h = rng.uniform(0.01, 0.05, cfg.channels).astype(np.float32)
    want = orc.state_passing(cfg, loc, gamma, init, s_h)
    buf = torch.zeros((chunks + 1) * per, device="cuda")
    dl = buf[per:]
    dl.copy_(gh.dev(loc).reshape(-1))
    dp = {None: None, "own": torch.empty_like(dl), "loc": dl, "before loc": buf[:-per]}[prev]
    fin, hq = torch.empty(init.shape, device="cuda"), torch.empty(loc.shape, dtype=torch.int8, device="cuda")
    bd.ssdi8_state_passing(bd.dims_of(cfg), dl, gh.dev(gamma), gh.dev(init), dp, fin, hq, gh.dev(s_h))
    torch.cuda.synchronize()
    assert prev is None or np.array_equal(dp.cpu().numpy(), np.asarray(want[0]).reshape(-1))
    assert np.array_equal(fin.cpu().numpy(), want[1]) and np.array_equal(hq.cpu().numpy(), want[2])


@pytest.mark.parametrize("b,H", [(1, 23), (1, 25), (2, 33)])
def test_state_passing_on_either_side_of_the_thread_limit(b, H):
    # 16 chunks: up to 98 304 threads (48 heads of 64 x 128 states) keep the next batch ahead
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("threads", b, 64 * 17, 2 * H, 64, 128, 1, 64, 0.02, 20.0, 49)
    rng = np.random.default_rng(H)
    loc = rng.standard_normal((b, 17, 2 * H, 64, 128)).astype(np.float32)
    gamma = rng.uniform(0, 1, (b, 2 * H, 17)).astype(np.float32)
    s_h = rng.uniform(0.01, 0.05, cfg.channels).astype(np.float32)
    want = orc.state_passing(cfg, loc, gamma, None, s_h)
    fin, hq = torch.empty((b, 2 * H, 64, 128), device="cuda"), torch.empty(loc.shape, dtype=torch.int8, device="cuda")
    bd.ssdi8_state_passing(bd.dims_of(cfg), gh.dev(loc), gh.dev(gamma), None, None, fin, hq, gh.dev(s_h))
    torch.cuda.synchronize()
    assert np.array_equal(fin.cpu().numpy(), want[1]) and np.array_equal(hq.cpu().numpy(), want[2])


def test_a_state_that_is_not_a_number_has_the_same_codes_on_both_state_routes():
    # 9 chunks take the two kernels, the same call with the INT8 state flag off and more heads the fused one: the codes of the
    # first chunk's entering state are those of init_state alone
    import gpu_harness as gh
    few = SSDConfig("few", 1, 9 * 64, 4, 64, 64, 1, 64, 0.02, 20.0, 50)
    many = SSDConfig("many", 1, 9 * 64, 160, 64, 64, 1, 64, 0.02, 20.0, 50)
    hq = []
    for cfg in (few, many):
        q = _random_codes(cfg, 50)
        q["init"][:] = 0.25
        q["init"][0, 1, 7, 3:9] = np.array([0x7fc00000, 0xffc00000, 0x7f800000, 0xff800000, 0x00000000, 0x80000000],
                                           np.uint32).view(np.float32)
        q["s_h"][64:66] = 0.0
        hq.append(gh.gpu_fwd(cfg, q, taps=("hq",))[2]["hq"][0, 0, :4])
    assert np.array_equal(hq[0], hq[1])


@pytest.mark.parametrize("N,Q", [(64, 64), (128, 256)])
def test_a_state_that_is_not_a_number_has_the_same_codes_in_a_cluster(N, Q):
    # Eight chunks of four heads take a cluster per head, the same heads among 160 the fused kernel: the codes of every chunk's entering
    # state and the final state are the same, also where a NaN or an infinity goes through all chunks
    import gpu_harness as gh
    many = SSDConfig("many", 1, 8 * Q, 160, 64, N, 1, Q, 0.02, 20.0, 75)
    few = SSDConfig("few", 1, 8 * Q, 4, 64, N, 1, Q, 0.02, 20.0, 75)
    q = _random_codes(many, 75)
    q["init"][0, 1, 7, 3:9] = np.array([0x7fc00000, 0xffc00000, 0x7f800000, 0xff800000, 0x00000000, 0x80000000], np.uint32).view(np.float32)
    q["s_h"][64:66] = 0.0
    q["A"][1] = -0.01   # (a decay of 0 would make NaNs of the infinities)
    r = dict(q, init=q["init"][:, :4], A=q["A"][:4], D=q["D"][:4], **{k: np.asarray(q[k]).reshape(8 * Q, 160, -1)[:, :4] for k in ("xq", "dt")},
             **{k: q[k][:256] for k in ("s_x", "s_xs", "s_h")})
    _, fin, got = gh.gpu_fwd(many, q, taps=("hq",))
    _, fin_few, got_few = gh.gpu_fwd(few, {k: np.ascontiguousarray(v) for k, v in r.items()}, taps=("hq",))
    assert np.isnan(fin[0, 1, 7, 3]) and np.isinf(fin[0, 1, 7, 5])
    assert np.array_equal(got_few["hq"], got["hq"][:, :, :4])
    assert np.array_equal(fin_few, fin[:, :4], equal_nan=True)


@pytest.mark.parametrize("b,c,H,N", [(1, 3, 5, 64), (2, 1, 150, 128)])
def test_calibration_passes_over_states_that_are_not_a_number(b, c, H, N):
    # A NaN in init_state counts for nothing in the step size of its channel, as one anywhere else does: the step sizes are
    # those with a zero in its place in every other channel, and finite in its own
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("cal_nan", b, c * 64, H, 64, N, 1, 64, 0.02, 20.0, 51)
    q = _random_codes(cfg, 51)
    at = ((0, 1, 7, 5), (b - 1, H - 1, 63, N - 1))
    s_h = []
    for bad in (0.0, np.nan):
        init = q["init"].copy()
        for i in at:
            init[i] = bad
        dv = {k: gh.dev(q[k]) for k in ("xq", "Bq", "Cq", "s_x", "s_B", "s_C", "dt", "A")}
        s = [torch.empty(n, device="cuda") for n in (H * 64, 1, H * 64)]
        bd.ssdi8_calibrate(bd.dims_of(cfg), bd.make_fwd_args(init_state=gh.dev(init), **dv), *s, bd.alloc_workspace(bd.dims_of(cfg)))
        s_h.append(s[2].cpu().numpy())
    own = np.zeros(H * 64, bool)
    own[[h * 64 + p for _, h, p, _ in at]] = True
    assert np.array_equal(s_h[0][~own], s_h[1][~own])
    assert np.all(np.isfinite(s_h[1])) and np.all(s_h[1][own] <= s_h[0][own]) and np.all(s_h[1][own] > 0)


def test_calibration_takes_slices_of_packed_step_sizes():
    # s_x, s_B, s_C, A and the outputs 4-byte aligned only
    import torch
    import gpu_harness as gh
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("cal_slices", 1, 3 * 128, 9, 64, 64, 3, 128, 0.02, 20.0, 52)
    q = _random_codes(cfg, 52)
    dims = bd.dims_of(cfg)
    HP, G = cfg.channels, cfg.ngroups
    dv = {k: gh.dev(q[k]) for k in ("xq", "Bq", "Cq", "s_x", "s_B", "s_C", "dt", "A")}
    dv["s_x"] = dv["s_x"] * torch.linspace(0.5, 2.0, HP, device="cuda")
    got = []
    for shift in (0, 1, 2, 3):
        put = lambda t: torch.cat([torch.zeros(shift, device="cuda"), t])[shift:]
        args = bd.make_fwd_args(**{k: put(v) if k in ("s_x", "s_B", "s_C", "A") else v for k, v in dv.items()})
        s = [torch.empty(n + shift, device="cuda")[shift:] for n in (HP, G, HP)]
        bd.ssdi8_calibrate(dims, args, *s, bd.alloc_workspace(dims))
        got.append(torch.cat(s).cpu().numpy())
    assert all(np.array_equal(g, got[0]) for g in got[1:])


def test_calibration_on_a_sequence_of_more_than_four_million_tokens():
    # s_xs and s_cb do not depend on how the chunks are shared out among batch elements
    import torch
    from paper_2608_21952_b200 import binding as bd
    g = torch.Generator(device="cuda").manual_seed(53)
    T = 256 * 5 * 3277
    i8 = lambda: torch.randint(-127, 128, (T, 64), generator=g, device="cuda", dtype=torch.int8)
    q = dict(xq=i8(), Bq=i8(), Cq=i8(), dt=0.01 + 0.1 * torch.rand(T, 1, generator=g, device="cuda"),
             A=torch.full((1,), -0.5, device="cuda"), s_x=0.01 + torch.rand(64, generator=g, device="cuda"),
             s_B=torch.full((1,), 0.03, device="cuda"), s_C=torch.full((1,), 0.03, device="cuda"))
    got = []
    for b in (1, 5):
        dims = bd.Dims(b, T // b, 1, 64, 64, 1, 256)
        s = [torch.empty(n, device="cuda") for n in (64, 1, 64)]
        ws = bd.alloc_workspace(dims)
        bd.ssdi8_calibrate(dims, bd.make_fwd_args(**q), *s, ws)
        got.append([t.cpu().numpy() for t in s])
        del ws
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    assert np.all(np.isfinite(got[0][2])) and np.all(got[0][2] > 0)


def test_host_pipeline_calls_from_several_threads():
    # each thread with its stream, scratch, buffers and inputs; slices in one piece per call and in many
    import threading
    import torch
    from paper_2608_21952_b200 import binding as bd

    def setup(seed, b, c, H):
        cfg = SSDConfig("threads", b, c * 128, H, 64, 64, 1, 128, 0.02, 20.0, seed)
        dims = bd.dims_of(cfg)
        g = torch.Generator().manual_seed(seed)
        T, HP = cfg.tokens, cfg.channels
        r = lambda *s: torch.randn(*s, generator=g)
        host = {"x": r(T, HP), "B": r(T, 64), "C": r(T, 64), "dt": torch.nn.functional.softplus(r(T, H) - 3.0)}
        host = {k: v.pin_memory() for k, v in host.items()}
        par = {"A": -torch.exp(r(H)), "D": r(H), "s_x": torch.full((HP,), 0.03), "s_B": torch.full((1,), 0.03),
               "s_C": torch.full((1,), 0.03), "s_xs": torch.full((HP,), 0.002), "s_cb": torch.full((1,), 0.4),
               "s_h": torch.full((HP,), 0.02)}
        par = {k: v.cuda() for k, v in par.items()}
        y, fin = torch.empty(T, HP, device="cuda"), torch.empty(b, H, 64, 64, device="cuda")
        ws = torch.empty(bd.ssdi8_layer_fwd_workspace_bytes(dims, 0), dtype=torch.uint8, device="cuda")
        bd.ssdi8_layer_fwd(dims, bd.make_layer_args(y=y, final_state=fin, **{k: v.cuda() for k, v in host.items()}, **par), ws)
        torch.cuda.synchronize()
        scratch = torch.empty(bd.ssdi8_layer_fwd_host_scratch_bytes(dims, 0), dtype=torch.uint8, device="cuda")
        return dims, host, par, scratch, y.cpu(), fin.cpu()

    work = [setup(60, 2, 12, 40), setup(61, 9, 1, 80), setup(62, 1, 9, 200)]
    wrong = []

    def run(dims, host, par, scratch, y, fin):
        try:
            stream = torch.cuda.Stream()
            for _ in range(8):
                yh = torch.full(y.shape, float("nan")).pin_memory()
                fh = torch.full(fin.shape, float("nan")).pin_memory()
                bd.ssdi8_layer_fwd_host(dims, bd.make_host_args(y=yh, final_state=fh, **host, **par), scratch, stream=stream)
                stream.synchronize()
                if not (torch.equal(yh, y) and torch.equal(fh, fin)):
                    wrong.append(dims.nheads)
        except BaseException as e:   # noqa: BLE001 (a thread's exception would not fail the test)
            wrong.append(e)

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def test_host_pipeline_that_ends_early_leaves_the_stream_behind_its_copies():
    # an initial state that is not 16-byte aligned is refused by the first slice's kernels, with the slice's copies on their way:
    # after the caller's stream they are complete
    import torch
    from paper_2608_21952_b200 import binding as bd
    cfg = SSDConfig("early", 1, 24 * 128, 80, 64, 64, 1, 128, 0.02, 20.0, 63)
    dims = bd.dims_of(cfg)
    T, HP = cfg.tokens, cfg.channels
    pin = lambda *s: torch.randn(*s).pin_memory()
    x, y = pin(T, HP), torch.empty(T, HP).pin_memory()
    c = lambda n: torch.ones(n, device="cuda")
    init = torch.zeros(80 * 64 * 64 + 1, device="cuda")[1:]
    scratch = torch.zeros(bd.ssdi8_layer_fwd_host_scratch_bytes(dims, 0), dtype=torch.uint8, device="cuda")
    args = bd.make_host_args(x=x, B=pin(T, 64), C=pin(T, 64), dt=torch.rand(T, 80).pin_memory(), A=-c(80), y=y, init_state=init,
                             s_x=c(HP), s_B=c(1), s_C=c(1), s_xs=c(HP), s_cb=c(1), s_h=c(HP))
    torch.cuda.synchronize()
    with pytest.raises(bd.SSDi8Error) as e:
        bd.ssdi8_layer_fwd_host(dims, args, scratch)
    first = scratch[:128 * HP * 4].clone()   # x of the first chunk, at the start of the scratch
    assert e.value.code == bd.ERR_ALIGN
    assert torch.equal(first.view(torch.float32).cpu(), x[:128].reshape(-1))
    args.init_state = 0
    bd.ssdi8_layer_fwd_host(dims, args, scratch)
    torch.cuda.synchronize()
    assert torch.isfinite(y).all()
