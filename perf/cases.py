"""The work that a user of this library has it do, as cases that can be timed and whose outputs can be compared.

Five kinds of call, all through the binding:

  layer      one SSD layer on fp32 x, B, C and a positive time step: `ssdi8_layer_fwd` (what bench.py steps)
  prefill    the same layer inside a 16-bit model: the convolution output xBC goes through `ssdi8_quantize_entry`,
             Algorithm 2 through `ssdi8_chunk_scan_fwd` from the raw time step, with the state and output format and
             the ChunkScan operand that the model was set up with
  decode     one token for every sequence: `ssdi8_quantize_entry` on one row per sequence, `ssdi8_softplus_dt`,
             `ssdi8_ssd_step` on the state in place
  calibrate  static step sizes from a sample batch: `ssdi8_quantize_act` (mode 1) on x, B and C, `ssdi8_calibrate`
  host       the layer from page-locked host buffers: `ssdi8_layer_fwd_host`

Shapes are those of paper_2608_21952_b200/inputs.py, the tests, or in between; the values follow the same recipe as
there (outlier channels in x, unit-scale B and C, softplus(N(-3, 1)) time steps, log-uniform decay rates).  The step
sizes are static, calibrated in `prepare` on the same tensors.
"""
import math

import torch

from paper_2608_21952_b200 import binding as bd

P = 64   # head dimension (the only one the library takes)


def _case(name, kind, batch, seqlen, nheads, dstate, ngroups, chunk, **options):
    c = {} if name is None else {"name": name}
    c.update({"kind": kind, "batch": batch, "seqlen": seqlen, "nheads": nheads, "dstate": dstate,
              "ngroups": ngroups, "chunk": chunk, "dtype": "float32", "y": "float32", "int8_state": False,
              "fp16_operand": False, "init": False, "corr": False})
    c.update(options)
    return c


def listed():
    return [
        # the smallest supported layer of the workload table: eight chunks of 64 tokens, latency and launches
        _case("layer 1x512x4", "layer", 1, 512, 4, 64, 1, 64),
        # the 130M-shaped layer on one sequence: a single user's prompt, fewer units than SMs
        _case("layer 1x2048x24", "layer", 1, 2048, 24, 128, 1, 256),
        # the 2.7B-shaped layer at batch 8: the workload of bench.py
        _case("layer 8x2048x80", "layer", 8, 2048, 80, 128, 1, 256),
        # the 8B-shaped layer with groups on long sequences: the largest
        _case("layer 4x8192x128", "layer", 4, 8192, 128, 128, 8, 256),
        # a ragged one: odd batch and chunk counts, 50 heads in two groups, the smaller state, chunks of 128
        _case("layer 3x1408x50", "layer", 3, 1408, 50, 64, 2, 128, y="bfloat16", corr=True),
        # a short prompt of one chunk in a bf16 model
        _case("prefill 1x256x24", "prefill", 1, 256, 24, 128, 1, 256, dtype="bfloat16", y="bfloat16"),
        # a serving batch in a bf16 model that goes on from cached states
        _case("prefill 5x1792x80", "prefill", 5, 1792, 80, 128, 1, 256, dtype="bfloat16", y="bfloat16", init=True),
        # the paper's own formats: INT8 states, FP16 ChunkScan operand, FP16 output, mean correction
        _case("prefill 8x2048x80 paper", "prefill", 8, 2048, 80, 128, 1, 256, dtype="float16", y="float16",
              int8_state=True, fp16_operand=True, corr=True),
        # decode of one sequence of the 130M shape: three short launches
        _case("decode 1x24", "decode", 1, 1, 24, 128, 1, 256, dtype="bfloat16"),
        # decode of a full batch of the 2.7B shape: the state is larger than L2
        _case("decode 64x80", "decode", 64, 1, 80, 128, 1, 256, dtype="bfloat16"),
        # offline calibration on a sample batch of the 2.7B shape
        _case("calibrate 2x2048x80", "calibrate", 2, 2048, 80, 128, 1, 256),
        # inputs and outputs in host memory
        _case("host 3x1024x80", "host", 3, 1024, 80, 128, 1, 256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "prefill", "prefill", "prefill", "decode", "decode", "calibrate", "host"])
    dstate = rng.choice([64, 128, 128])
    ngroups = rng.choice([1, 1, 1, 2, 4, 8])
    nheads = ngroups * max(1, _log_int(rng, 4, 128) // ngroups)
    dtype = rng.choice(["bfloat16", "bfloat16", "float16"])
    if kind == "decode":
        return _case(None, kind, _log_int(rng, 1, 96), 1, nheads, dstate, ngroups, 256, dtype=dtype, corr=rng.random() < 0.3)
    chunk = rng.choice([64, 128, 256, 256])
    # total tokens x heads, from the smallest listed layer to half the largest, spread over the logarithm
    most = {"layer": 2 << 20, "prefill": 2 << 20, "calibrate": 1 << 19, "host": 1 << 19}[kind]
    tokens = max(chunk, _log_int(rng, 2048, most) // nheads)
    batch = max(1, min(_log_int(rng, 1, 12), tokens // chunk))
    seqlen = chunk * max(1, min(tokens // batch // chunk, 8192 // chunk))
    y = rng.choice(["float32", "float32", "bfloat16", "float16"])
    c = _case(None, kind, batch, seqlen, nheads, dstate, ngroups, chunk, y=y, corr=rng.random() < 0.3,
              int8_state=rng.random() < 0.25, fp16_operand=rng.random() < 0.25)
    if kind == "prefill":
        c.update(dtype=dtype, init=rng.random() < 0.5)
    if kind == "calibrate":
        c.update(y="float32", corr=False, int8_state=False, fp16_operand=False)
    return c


def _flags(case):
    f = {"float32": 0, "float16": bd.FLAG_Y_FP16, "bfloat16": bd.FLAG_Y_BF16}[case["y"]]
    if case["int8_state"]:
        f |= bd.FLAG_INT8_STATE
    if case["fp16_operand"]:
        f |= bd.FLAG_FP16_OPERAND
    return f


def _static_scales(dims, x, B, C, dt, A, init):
    """Step sizes of x, B, C and of the internal tensors, calibrated on the given tensors."""
    T, G = dims.batch * dims.seqlen, dims.ngroups
    HP = dims.nheads * P
    new = lambda n: torch.empty(n, device="cuda")  # noqa: E731
    s = {"s_x": new(HP), "s_B": new(G), "s_C": new(G), "s_xs": new(HP), "s_cb": new(G), "s_h": new(HP)}
    q = {"xq": torch.empty(x.shape, dtype=torch.int8, device="cuda"),
         "Bq": torch.empty(B.shape, dtype=torch.int8, device="cuda"),
         "Cq": torch.empty(C.shape, dtype=torch.int8, device="cuda")}
    bd.ssdi8_quantize_act(x, T, HP, 1, s["s_x"], 1, q["xq"])
    bd.ssdi8_quantize_act(B, T, G, dims.dstate, s["s_B"], 1, q["Bq"])
    bd.ssdi8_quantize_act(C, T, G, dims.dstate, s["s_C"], 1, q["Cq"])
    args = bd.make_fwd_args(dt=dt, A=A, init_state=init, s_x=s["s_x"], s_B=s["s_B"], s_C=s["s_C"], **q)
    bd.ssdi8_calibrate(dims, args, s["s_xs"], s["s_cb"], s["s_h"], bd.alloc_workspace(dims))
    return s


def prepare(case, seed):
    b, L, H, N, G, kind = (case["batch"], case["seqlen"], case["nheads"], case["dstate"], case["ngroups"], case["kind"])
    g = torch.Generator(device="cuda").manual_seed(seed)
    randn = lambda *shape: torch.randn(shape, generator=g, device="cuda")  # noqa: E731
    T, HP = b * L, H * P
    x = randn(T, HP)
    x[:, torch.randperm(HP, generator=g, device="cuda")[:math.ceil(0.01 * HP)]] *= 50.0
    B, C = randn(T, G * N), randn(T, G * N)
    A = -torch.exp(torch.rand(H, generator=g, device="cuda") * math.log(16.0))
    D = randn(H)
    dt_bias = torch.full((H,), -3.0, device="cuda") + 0.25 * randn(H)
    dt_raw = randn(T, H)
    dt = torch.nn.functional.softplus(dt_raw + dt_bias)
    corr = 0.01 * randn(HP) if case["corr"] else None
    dtype = getattr(torch, case["dtype"])
    xBC = torch.cat([x, B, C], dim=1).to(dtype).contiguous() if kind in ("prefill", "decode") else None
    dims = bd.Dims(b, L, H, P, N, G, case["chunk"])
    st = {"case": case, "dims": dims}
    codes = {"xq": torch.empty(T, HP, dtype=torch.int8, device="cuda"),
             "Bq": torch.empty(T, G * N, dtype=torch.int8, device="cuda"),
             "Cq": torch.empty(T, G * N, dtype=torch.int8, device="cuda")}

    if kind == "calibrate":
        new = lambda n: torch.empty(n, device="cuda")  # noqa: E731
        st["in"] = {"x": x, "B": B, "C": C}
        st["scales"] = {"s_x": new(HP), "s_B": new(G), "s_C": new(G), "s_xs": new(HP), "s_cb": new(G), "s_h": new(HP)}
        st["codes"] = codes
        s = st["scales"]
        st["args"] = bd.make_fwd_args(dt=dt, A=A, s_x=s["s_x"], s_B=s["s_B"], s_C=s["s_C"], **codes)
        st["ws"] = bd.alloc_workspace(dims)
        return st

    if kind == "decode":
        absmax = lambda t: t.abs().amax(dim=0) / 127.0  # noqa: E731
        st.update(xBC=xBC, codes=codes, dt_raw=dt_raw, dt_bias=dt_bias, A=A, D=D, corr=corr,
                  # (one row per sequence: per-channel step sizes of a batch this small would depend on the batch alone)
                  s_x=torch.clamp(absmax(x), min=0.02), s_B=torch.full((G,), 4.0 / 127.0, device="cuda"),
                  s_C=torch.full((G,), 4.0 / 127.0, device="cuda"), dt=torch.empty_like(dt_raw),
                  state=randn(b, H, P, N), y_out=torch.empty(b, H, P, device="cuda"))
        return st

    y_dtype = getattr(torch, case["y"])
    init = randn(b, H, P, N) if case["init"] else None
    if kind == "prefill":
        xc, Bc, Cc = (t.float().contiguous() for t in xBC.split([HP, G * N, G * N], dim=1))
    else:
        xc, Bc, Cc = x, B, C
    s = _static_scales(dims, xc, Bc, Cc, dt, A, init)
    flags = _flags(case)
    if kind == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        st["y_out"] = torch.empty(b, L, H, P, dtype=y_dtype).pin_memory()
        st["fin"] = torch.empty(b, H, P, N).pin_memory()
        st["args"] = bd.make_host_args(x=pin(x), B=pin(B), C=pin(C), dt=pin(dt), A=A, D=D, corr=corr, y=st["y_out"],
                                       final_state=st["fin"], status=torch.zeros(1, dtype=torch.int32).pin_memory(), **s)
        st["ws"] = torch.empty(bd.ssdi8_layer_fwd_host_scratch_bytes(dims, flags), dtype=torch.uint8, device="cuda")
        st["flags"] = flags
        return st
    st["y_out"] = torch.empty(b, L, H, P, dtype=y_dtype, device="cuda")
    st["fin"] = torch.empty(b, H, P, N, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    if kind == "layer":
        st["args"] = bd.make_layer_args(x=x, B=B, C=C, dt=dt, A=A, D=D, corr=corr, y=st["y_out"], final_state=st["fin"],
                                        status=status, **s)
        st["ws"] = torch.empty(bd.ssdi8_layer_fwd_workspace_bytes(dims, flags), dtype=torch.uint8, device="cuda")
    else:
        flags |= bd.FLAG_DT_SOFTPLUS
        st.update(xBC=xBC, codes=codes, s=s)
        st["args"] = bd.make_fwd_args(dt=dt_raw, dt_bias=dt_bias, A=A, D=D, corr=corr, init_state=init, y=st["y_out"],
                                      final_state=st["fin"], status=status, **codes, **s)
        st["ws"] = bd.alloc_workspace(dims, flags=flags)
    st["flags"] = flags
    return st


def run(st):
    case, dims = st["case"], st["dims"]
    kind, T, HP, G, N = case["kind"], case["batch"] * case["seqlen"], case["nheads"] * P, case["ngroups"], case["dstate"]
    if kind == "layer":
        bd.ssdi8_layer_fwd(dims, st["args"], st["ws"], flags=st["flags"])
        return {"y": st["y_out"], "final_state": st["fin"]}
    if kind == "host":
        # (returns once everything is enqueued; the buffers are complete when the stream has been waited for)
        bd.ssdi8_layer_fwd_host(dims, st["args"], st["ws"], flags=st["flags"])
        return {"y": st["y_out"], "final_state": st["fin"]}
    if kind == "prefill":
        q, s = st["codes"], st["s"]
        bd.ssdi8_quantize_entry(st["xBC"], T, HP, G, N, s["s_x"], s["s_B"], s["s_C"], q["xq"], q["Bq"], q["Cq"])
        bd.ssdi8_chunk_scan_fwd(dims, st["args"], st["ws"], flags=st["flags"])
        return {"y": st["y_out"], "final_state": st["fin"]}
    if kind == "decode":
        q = st["codes"]
        bd.ssdi8_quantize_entry(st["xBC"], T, HP, G, N, st["s_x"], st["s_B"], st["s_C"], q["xq"], q["Bq"], q["Cq"])
        bd.ssdi8_softplus_dt(st["dt_raw"], st["dt_bias"], T, case["nheads"], st["dt"])
        bd.ssdi8_ssd_step(dims, q["xq"], st["s_x"], q["Bq"], st["s_B"], q["Cq"], st["s_C"], st["dt"], st["A"], st["D"],
                          st["corr"], st["state"], st["y_out"])
        return {"y": st["y_out"], "state": st["state"]}
    t, q, s = st["in"], st["codes"], st["scales"]
    bd.ssdi8_quantize_act(t["x"], T, HP, 1, s["s_x"], 1, q["xq"])
    bd.ssdi8_quantize_act(t["B"], T, G, N, s["s_B"], 1, q["Bq"])
    bd.ssdi8_quantize_act(t["C"], T, G, N, s["s_C"], 1, q["Cq"])
    bd.ssdi8_calibrate(dims, st["args"], s["s_xs"], s["s_cb"], s["s_h"], st["ws"])
    return {**q, **s}


def work(case):
    """Inputs read once and outputs written once; two operations per multiply-accumulate of the contractions (the causal
    half of the square ones)."""
    b, L, H, N, G, Q = (case["batch"], case["seqlen"], case["nheads"], case["dstate"], case["ngroups"], case["chunk"])
    kind, T = case["kind"], case["batch"] * case["seqlen"]
    size = {"float32": 4, "float16": 2, "bfloat16": 2}
    state = b * H * P * N * 4
    row = H * P + 2 * G * N
    if kind == "decode":
        return {"bytes": T * row * size[case["dtype"]] + T * H * 4 + 2 * state + T * H * P * 4, "flops": 5.0 * T * H * P * N}
    contractions = 2.0 * T * (G * N * (Q + 1) / 2 + 2 * H * P * N + H * P * (Q + 1) / 2)   # C B^T; B^T x and C h; (L o C B^T) x
    if kind == "calibrate":
        return {"bytes": T * row * 5 + T * H * 4, "flops": 2.0 * T * (G * N * (Q + 1) / 2 + H * P * N)}
    moved = T * row * size[case["dtype"]] + T * H * 4 + T * H * P * size[case["y"]] + state * (2 if case["init"] else 1)
    return {"bytes": moved, "flops": contractions}


def tolerance(case):
    """About four times what one rounding of the time step (a relative 6e-8) changes, measured over the listed cases and
    fourteen drawn ones: another exponential or another order of a sum moves the codes of the internal int8 tensors that
    lie next to a rounding boundary, and one code moves its row of y (rel 1.7e-4, max 0.21; 7.2e-4 and 0.29 where the
    states are int8 codes too).  Decode and calibration hold binary32 sums only (rel 9.3e-8, max 3.1e-6; rel 3.7e-7, max
    5.2e-6); the codes of x, B and C are the same numbers in any correct implementation."""
    if case["kind"] == "calibrate":
        return {"rel": 1.5e-6, "max": 2e-5}
    if case["kind"] == "decode":
        return {"rel": 4e-7, "max": 1.2e-5}
    return {"rel": 3e-3, "max": 0.9} if case["int8_state"] else {"rel": 7e-4, "max": 0.8}
