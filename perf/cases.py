"""The work a program gives this library, as measurable cases: tensors converted to HiF8 and back, fake-quantized tensors,
matrix products on HiF8 operands, and the training step of one linear layer.

A case is a dict of plain values.  `kind` names the sequence of calls; the sizes, the source format, the rounding method and
the operand layouts are the rest of it.  Inputs are drawn on the GPU from the case's seed: bell-shaped activations and
weights (a few channels of an activation carry outliers), log-uniform gradients.
"""
import torch

import paper_2409_16626_b200 as H

TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
HIF8 = {"f32": H.F32, "bf16": H.BF16, "f16": H.F16}
SIZE = {"f32": 4, "bf16": 2, "f16": 2}
RND = {"ta": H.RND_TA, "hr": H.RND_HR, "ssr": H.RND_SSR}

LARGEST_GEMM = 8192 * 28672 * 8192
LARGEST_TENSOR = 1 << 28


def listed():
    return [
        # the activations of sixteen decoded tokens, quantized in front of a layer: latency and launches
        {"name": "scale_encode_tokens", "kind": "scale_encode", "n": 16 * 8192, "dtype": "bf16", "rnd": "ta", "values": "normal"},
        # one optimizer's view of a weight or activation tensor: scaled to HiF8 and back in FP32
        {"name": "roundtrip_f32", "kind": "roundtrip", "n": 4096 * 4096, "dtype": "f32", "rnd": "ta", "values": "normal"},
        # simulated quantization of a block of activations with outlier channels, as in a quantization-aware run
        {"name": "fake_quant_bf16", "kind": "fake_quant", "n": 8192 * 8192, "dtype": "bf16", "rnd": "hr", "values": "outliers"},
        # the largest conversion: a gradient bucket of wide dynamic range, hybrid rounding, a scale known beforehand
        {"name": "encode_gradient", "kind": "encode", "n": 1 << 28, "dtype": "f32", "rnd": "hr", "values": "loguniform"},
        # a checkpoint shard of odd length read back into BF16
        {"name": "decode_shard", "kind": "decode", "n": 3001 * 4099, "dtype": "bf16", "rnd": "ta", "values": "normal"},
        # a layer's weight converted once with one scale per output channel
        {"name": "channel_weights", "kind": "channel_encode", "rows": 7168, "cols": 4096, "axis": 0, "dtype": "bf16", "rnd": "ta"},
        # inference, decode phase: sixteen tokens against a large weight
        {"name": "gemm_decode", "kind": "gemm", "m": 16, "n": 28672, "k": 8192, "layout": "nk", "out": "bf16", "channel": False, "workspace": "full"},
        # inference, a batch of short prompts of ragged total length, one scale per weight channel
        {"name": "gemm_batch", "kind": "gemm", "m": 201, "n": 7168, "k": 4096, "layout": "nk", "out": "bf16", "channel": True, "workspace": "full"},
        # prefill of a long prompt, the largest product
        {"name": "gemm_prefill", "kind": "gemm", "m": 8192, "n": 28672, "k": 8192, "layout": "kn", "out": "bf16", "channel": False, "workspace": "full"},
        # the same kind of product where the caller has no memory to spare beyond the status word
        {"name": "gemm_no_workspace", "kind": "gemm", "m": 2048, "n": 7168, "k": 4096, "layout": "kn", "out": "bf16", "channel": False, "workspace": "status"},
        # a training step of one linear layer: three conversions, forward, both backward products, two micro-batches
        {"name": "linear_step", "kind": "linear_step", "tokens": 2048, "fan_in": 4096, "fan_out": 7168},
        # the same for a small layer, where launches count
        {"name": "linear_step_small", "kind": "linear_step", "tokens": 256, "fan_in": 768, "fan_out": 1536},
    ]


def _log(rng, lo, hi, step=1):
    """A size between lo and hi, spread over its logarithm, a multiple of `step`."""
    v = lo * (hi / lo) ** rng.random()
    return max(lo, min(hi, int(v) // step * step))


def draw(rng):
    kind = rng.choice(["scale_encode", "roundtrip", "fake_quant", "encode", "decode", "channel_encode", "gemm", "gemm", "gemm", "gemm", "linear_step", "linear_step"])
    if kind == "gemm":
        while True:
            c = {"kind": kind, "m": _log(rng, 1, 8192), "n": _log(rng, 512, 28672, 16), "k": _log(rng, 512, 16384, 16),
                 "layout": rng.choice(["nk", "kn"]), "out": rng.choice(["bf16", "bf16", "f32"]), "channel": rng.random() < 0.3,
                 "workspace": rng.choice(["full", "full", "full", "status"])}
            if c["m"] * c["n"] * c["k"] <= LARGEST_GEMM // (4 if c["workspace"] == "status" else 1):
                return c
    if kind == "linear_step":
        return {"kind": kind, "tokens": _log(rng, 64, 4096, 16), "fan_in": _log(rng, 512, 8192, 16), "fan_out": _log(rng, 512, 8192, 16)}
    if kind == "channel_encode":
        return {"kind": kind, "rows": _log(rng, 256, 28672, 8), "cols": _log(rng, 256, 8192, 8), "axis": rng.choice([0, 1]),
                "dtype": rng.choice(["bf16", "f32"]), "rnd": "ta"}
    n = _log(rng, 512, LARGEST_TENSOR // 2)
    if kind in ("scale_encode", "roundtrip"):
        return {"kind": kind, "n": n, "dtype": rng.choice(["bf16", "f32", "f16"]), "rnd": rng.choice(["ta", "hr"]), "values": rng.choice(["normal", "outliers"])}
    if kind == "fake_quant":
        return {"kind": kind, "n": n, "dtype": rng.choice(["bf16", "f32"]), "rnd": rng.choice(["ta", "hr"]), "values": rng.choice(["normal", "outliers"])}
    if kind == "encode":
        return {"kind": kind, "n": n, "dtype": rng.choice(["bf16", "f32"]), "rnd": rng.choice(["hr", "ssr", "ta"]), "values": "loguniform"}
    return {"kind": "decode", "n": n, "dtype": rng.choice(["bf16", "f16", "f32"]), "rnd": "ta", "values": "normal"}


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _values(n, dtype, values, g):
    """n elements: N(0,1); the same with every 1024th element times 100 (outlier channels); or signs and exponents in
    [-40, 20) uniform, as gradients with a wide dynamic range have them."""
    if values == "loguniform":
        e = torch.randint(127 - 40, 127 + 20, (n,), generator=g, device="cuda", dtype=torch.int32)
        x = e.bitwise_left_shift_(23).bitwise_or_(torch.randint(0, 1 << 23, (n,), generator=g, device="cuda", dtype=torch.int32)).view(torch.float32)
        x = torch.where(torch.randint(0, 2, (n,), generator=g, device="cuda", dtype=torch.uint8) > 0, x, -x)
    else:
        x = torch.randn(n, generator=g, device="cuda")
        if values == "outliers":
            x[::1024] *= 100
    return x.to(TORCH[dtype])


def _bytes(n):
    return torch.empty(n, dtype=torch.uint8, device="cuda")


def _scalars():
    return torch.zeros(1, dtype=torch.float32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.float32, device="cuda")


def _quantized(shape, std, g):
    """A BF16 tensor of that spread, converted by the library: its bytes and its scale exponent on the device."""
    n = shape[0] * shape[1]
    x = (torch.randn(n, generator=g, device="cuda") * std).bfloat16()
    q, (_, exp, _) = _bytes(n).view(shape), _scalars()
    ws = _bytes(H.hif8_workspace_bytes(H.WS_AMAX_SCALE_ENCODE, n))
    H.hif8_amax_scale_encode(x, H.BF16, q, n, d_scale_exp_out=exp, workspace=ws, workspace_bytes=ws.numel())
    return q, exp


def _prepare_gemm(c, g):
    m, n, k = c["m"], c["n"], c["k"]
    s = {"case": c}
    s["a"], s["sa"] = _quantized((m, k), 1.0, g)
    if c["channel"]:
        w = torch.randn(n * k, generator=g, device="cuda").mul_(0.02).bfloat16()
        shape = (n, k) if c["layout"] == "nk" else (k, n)
        s["w"], s["sw"] = _bytes(n * k).view(shape), torch.zeros(n, dtype=torch.int32, device="cuda")
        amax = torch.zeros(n, dtype=torch.float32, device="cuda")
        H.hif8_channel_amax_scale_encode(w, H.BF16, s["w"], shape[0], shape[1], 0 if c["layout"] == "nk" else 1, d_amax=amax, d_scale_exp_out=s["sw"])
    else:
        s["w"], s["sw"] = _quantized((n, k) if c["layout"] == "nk" else (k, n), 0.02, g)
    s["c"] = torch.empty(m, n, dtype=TORCH[c["out"]], device="cuda")
    s["ws"] = _bytes(H.hif8_workspace_bytes(H.WS_GEMM, m * k + k * n if c["workspace"] == "full" else 0))
    return s


def _prepare_step(c, g):
    t, i, o = c["tokens"], c["fan_in"], c["fan_out"]
    s = {"case": c, "x": [], "dy": []}
    for _ in range(2):
        s["x"].append(_values(t * i, "bf16", "outliers", g).view(t, i))
        s["dy"].append((torch.randn(t * o, generator=g, device="cuda") * torch.exp2(torch.randint(-12, 0, (t * o,), generator=g, device="cuda").float())).bfloat16().view(t, o))
    s["w"] = torch.randn(i * o, generator=g, device="cuda").mul_(0.02).bfloat16().view(i, o)
    s["xq"], s["wq"], s["dyq"] = _bytes(t * i).view(t, i), _bytes(i * o).view(i, o), _bytes(t * o).view(t, o)
    s["y"] = [torch.empty(t, o, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    s["dx"] = [torch.empty(t, i, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    s["dw"] = torch.empty(i, o, dtype=torch.float32, device="cuda")
    # delayed scaling of activations and gradients: the state a training program carries from step to step, already measured
    s["x_state"], s["dy_state"] = _bytes(H.SCALE_STATE_BYTES), _bytes(H.SCALE_STATE_BYTES)
    for state, src, dst in ((s["x_state"], s["x"][0], s["xq"]), (s["dy_state"], s["dy"][0], s["dyq"])):
        H.hif8_scale_state_init(state, 1)
        H.hif8_delayed_scale_encode(src, H.BF16, dst, src.numel(), H.RND_TA, 0, 0, state, 1)
    _, s["sw"], _ = _scalars()
    s["conv_ws"] = _bytes(H.hif8_workspace_bytes(H.WS_AMAX_SCALE_ENCODE, i * o))
    s["ws"] = _bytes(H.hif8_workspace_bytes(H.WS_GEMM, max(t * i + i * o, t * o + i * o, t * i + t * o)))
    return s


def prepare(case, seed):
    g, c, kind = _generator(seed), case, case["kind"]
    if kind == "gemm":
        return _prepare_gemm(c, g)
    if kind == "linear_step":
        return _prepare_step(c, g)
    s = {"case": c}
    n = c["rows"] * c["cols"] if kind == "channel_encode" else c["n"]
    x = _values(n, c["dtype"], c.get("values", "normal"), g)
    s["codes"] = _bytes(n)
    s["amax"], s["exp"], s["scale"] = _scalars()
    s["ws"] = _bytes(H.hif8_workspace_bytes(H.WS_AMAX_SCALE_ENCODE, n))
    if kind == "channel_encode":
        channels = c["rows"] if c["axis"] == 0 else c["cols"]
        s["amax"], s["exp"] = torch.zeros(channels, dtype=torch.float32, device="cuda"), torch.zeros(channels, dtype=torch.int32, device="cuda")
    if kind == "decode":
        H.hif8_amax_scale_encode(x, HIF8[c["dtype"]], s["codes"], n, workspace=s["ws"], workspace_bytes=s["ws"].numel(), d_scale_exp_out=s["exp"])
        s["scale_exp"] = int(s["exp"].item())
    else:
        s["x"] = x
    if kind in ("decode", "roundtrip", "fake_quant"):
        s["back"] = torch.empty(n, dtype=TORCH[c["dtype"]], device="cuda")
    return s


def _run_step(s):
    """One optimizer step's worth of a linear layer Y = X W: the weight converted once, then for each of two micro-batches
    forward, dX = dY W^T and dW += X^T dY; the gradient's amax is measured in the second conversion."""
    c = s["case"]
    t, i, o = c["tokens"], c["fan_in"], c["fan_out"]
    ws, wsb = s["ws"], s["ws"].numel()
    sx, sdy = s["x_state"], s["dy_state"]  # (the first int of a state is the exponent in force)
    H.hif8_amax_scale_encode(s["w"], H.BF16, s["wq"], i * o, d_scale_exp_out=s["sw"], workspace=s["conv_ws"], workspace_bytes=s["conv_ws"].numel())
    for b in range(2):
        H.hif8_delayed_scale_encode(s["x"][b], H.BF16, s["xq"], t * i, H.RND_TA, 0, 0, sx, 0)
        H.hif8_gemm(s["xq"], i, s["wq"], o, 0, s["y"][b], o, H.BF16, t, o, i, sx, s["sw"], ws, wsb)
        H.hif8_delayed_scale_encode(s["dy"][b], H.BF16, s["dyq"], t * o, H.RND_HR, 0, 0, sdy, 0)
        H.hif8_gemm_ex(s["dyq"], o, 0, s["wq"], o, 1, s["dx"][b], i, H.BF16, t, i, o, sdy, s["sw"], None, 0, ws, wsb)
        H.hif8_gemm_ex(s["xq"], i, 1, s["dyq"], o, 0, s["dw"], o, H.F32, i, o, t, sx, sdy, None, b, ws, wsb)
    return {"y": s["y"], "dx": s["dx"], "dw": s["dw"]}


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "linear_step":
        return _run_step(s)
    ws, wsb = s["ws"], s["ws"].numel()
    if kind == "gemm":
        m, n, k, nk = c["m"], c["n"], c["k"], int(c["layout"] == "nk")
        call = H.hif8_gemm_channel_scaled if c["channel"] else H.hif8_gemm
        call(s["a"], k, s["w"], k if nk else n, nk, s["c"], n, HIF8[c["out"]], m, n, k, s["sa"], s["sw"], ws, wsb)
        return s["c"]
    dt = HIF8[c["dtype"]]
    if kind == "channel_encode":
        H.hif8_channel_amax_scale_encode(s["x"], dt, s["codes"], c["rows"], c["cols"], c["axis"], 14, RND[c["rnd"]], d_amax=s["amax"], d_scale_exp_out=s["exp"])
        return [s["codes"], s["amax"], s["exp"]]
    n, rnd = c["n"], RND[c["rnd"]]
    if kind == "scale_encode":
        H.hif8_amax_scale_encode(s["x"], dt, s["codes"], n, 14, rnd, 0, 0, None, s["amax"], s["exp"], s["scale"], ws, wsb)
        return [s["codes"], s["amax"], s["exp"], s["scale"]]
    if kind == "roundtrip":
        H.hif8_amax_scale_encode(s["x"], dt, s["codes"], n, 14, rnd, 0, 0, None, s["amax"], s["exp"], s["scale"], ws, wsb)
        H.hif8_decode(s["codes"], s["back"], dt, n, 0)  # the scaled values; the exponent stays on the device
        return [s["codes"], s["back"], s["amax"], s["exp"], s["scale"]]
    if kind == "fake_quant":
        H.hif8_fake_quant(s["x"], s["back"], dt, n, 1, 14, rnd, 0, 0, s["amax"], s["exp"], ws, wsb)
        return [s["back"], s["amax"], s["exp"]]
    if kind == "encode":
        H.hif8_encode(s["x"], dt, s["codes"], n, 0, rnd)
        return s["codes"]
    H.hif8_decode(s["codes"], s["back"], dt, n, s["scale_exp"])
    return s["back"]


def work(case):
    c, kind = case, case["kind"]
    if kind == "gemm":
        m, n, k = c["m"], c["n"], c["k"]
        return {"bytes": m * k + n * k + m * n * SIZE[c["out"]], "flops": 2 * m * n * k}
    if kind == "linear_step":
        t, i, o = c["tokens"], c["fan_in"], c["fan_out"]
        # X, dY and W read as BF16; Y, dX and dW (FP32) written
        return {"bytes": 2 * (2 * t * i + 2 * t * o) + 2 * i * o + 2 * (2 * t * o + 2 * t * i) + 4 * i * o, "flops": 2 * 3 * 2 * t * i * o}
    n = c["rows"] * c["cols"] if kind == "channel_encode" else c["n"]
    size = SIZE[c["dtype"]]
    per = {"scale_encode": size + 1, "encode": size + 1, "decode": size + 1, "channel_encode": size + 1, "fake_quant": 2 * size, "roundtrip": 2 * size + 1}[kind]
    return {"bytes": n * per, "flops": 0}


def tolerance(case):
    kind = case["kind"]
    if kind not in ("gemm", "linear_step"):
        return "exact"  # every conversion is bit-exact, the dequantized values included
    # four times what the products show against the same products in 64 bits: 4.5e-7 and 2.5e-6 with FP32 results (K up to
    # 16384), 1.66e-3 and 3.9e-3 (half a unit in the last place and a little more) with BF16 results
    if kind == "gemm" and case["out"] == "f32":
        return {"rel": 2e-6, "max": 1e-5}
    return {"rel": 6.6e-3, "max": 1.6e-2}
