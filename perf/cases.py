"""Timed work of the nested-precision linear layers, one pass per case, through the public calls of the package.

Kinds of work (`case["kind"]`):

* ``single``   one small linear layer called eagerly, once in each mode: latency, launches and host work count.
* ``step``     a decoder step: the four linears (QKV, O, gate/up, down) of `layers` layers, each with weights and
               activations of its own, captured once as a CUDA graph per (tokens, mode) as a serving loop keeps it,
               and replayed.
* ``prefill``  the four linears of one layer on a prompt's tokens, called eagerly.
* ``fp8act``   the same layer in fast mode with FP8 activations: quantisation, then the FP8 linear, four times.
* ``moe``      one mixture-of-experts feed-forward: gate/up on rows gathered by token, then down on the expert rows,
               top-2 routing, encodings per expert, the caller keeps the workspace.
* ``load``     model loading: a layer's FP16 weights are split into planes (the encoding chosen from the data) and,
               as the check a loader makes, rebuilt.

Weights are FP16 0.02 * N(0, 1), activations FP16 N(0, 1); a tensor with `outliers` has a few weights of 2 to 6 at random
places, which is what makes the choice of the encoding fall on E5M2.
"""
import math

import torch

import paper_2609_34380_b200 as dps

MODES = {"fast": dps.DPS_MODE_FAST, "full": dps.DPS_MODE_FULL}
ENCODINGS = {"e4m3": dps.DPS_ENC_E4M3, "e5m2": dps.DPS_ENC_E5M2, "e4m3_rn": dps.DPS_ENC_E4M3_RN, "e5m2_rn": dps.DPS_ENC_E5M2_RN}

# rows of QKV, hidden and feed-forward sizes of the decoder layers
DECODER_4096 = {"hidden": 4096, "qkv": 12288, "ffn": 11008}
DECODER_8192 = {"hidden": 8192, "qkv": 10240, "ffn": 28672}
# the largest passes: 8192 tokens on a 4096-wide layer; weights of the 8192-wide layer twice
MAX_FLOPS = 2.0 * 8192 * 4096 * (12288 + 4096 + 3 * 11008)
MAX_STEP_WEIGHTS = 2 * 8192 * (10240 + 8192 + 3 * 28672)


def listed():
    return [
        # one 512 x 512 layer, 4 tokens: the smallest call a user makes
        {"name": "single_512_m4", "kind": "single", "n": 512, "k": 512, "tokens": 4, "enc": "e4m3"},
        # one user decoding
        {"name": "step_m1_fast", "kind": "step", "tokens": 1, "mode": "fast", "enc": "e4m3", "layers": 4, **DECODER_4096},
        # a small batch at full precision, a larger one in a burst
        {"name": "step_m8_full", "kind": "step", "tokens": 8, "mode": "full", "enc": "e4m3", "layers": 4, **DECODER_4096},
        {"name": "step_m32_fast", "kind": "step", "tokens": 32, "mode": "fast", "enc": "e4m3", "layers": 4, **DECODER_4096},
        # a batch and sizes that divide nothing evenly; weights out of E4M3 range
        {"name": "step_m13_full_ragged", "kind": "step", "tokens": 13, "mode": "full", "enc": "e5m2", "layers": 6,
         "hidden": 3088, "qkv": 4632, "ffn": 8336},
        # wide layers under load
        {"name": "step_m64_full_wide", "kind": "step", "tokens": 64, "mode": "full", "enc": "e4m3", "layers": 2, **DECODER_8192},
        {"name": "step_m256_fast_wide", "kind": "step", "tokens": 256, "mode": "fast", "enc": "e4m3", "layers": 1, **DECODER_8192},
        # a short prompt during a burst, a long one at full precision (the largest work)
        {"name": "prefill_m512_fast", "kind": "prefill", "tokens": 512, "mode": "fast", "enc": "e4m3", **DECODER_4096},
        {"name": "prefill_m8192_full", "kind": "prefill", "tokens": 8192, "mode": "full", "enc": "e4m3", **DECODER_4096},
        # a prompt of an odd length on the FP8 tensor cores
        {"name": "fp8act_m2999", "kind": "fp8act", "tokens": 2999, "enc": "e4m3", **DECODER_4096},
        # 256 tokens, two of eight experts each
        {"name": "moe_t256_fast", "kind": "moe", "tokens": 256, "mode": "fast", "experts": 8, "hidden": 4096, "ffn": 14336},
        # loading one layer
        {"name": "load_layer", "kind": "load", "outliers": 0, **DECODER_4096},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, lo, hi, step):
    return min(hi, max(lo, int(round(_log(rng, lo, hi) / step)) * step))


def _layer(rng, hidden_hi=8192):
    """Sizes of a decoder layer: one of the two above, or generic ones (hidden in 16s, QKV rows in 8s, grouped or not)."""
    if rng.random() < 0.4:
        return dict(DECODER_4096)
    if hidden_hi >= 8192 and rng.random() < 0.3:
        return dict(DECODER_8192)
    hidden = _size(rng, 512, hidden_hi, 16)
    return {"hidden": hidden, "qkv": 8 * int(hidden * rng.uniform(1.25, 3.0) / 8), "ffn": 16 * int(hidden * rng.uniform(2.5, 3.6) / 16)}


def _layer_weights(c):
    return c["hidden"] * (c["qkv"] + c["hidden"] + 3 * c["ffn"])


def draw(rng):
    kind = rng.choice(["single", "step", "step", "step", "step", "prefill", "prefill", "fp8act", "moe", "moe", "load"])
    mode = rng.choice(["fast", "full"])
    enc = rng.choice(["e4m3", "e4m3", "e4m3", "e5m2", "e4m3_rn", "e5m2_rn"])
    if kind == "single":
        return {"kind": kind, "n": _size(rng, 256, 4096, 8), "k": _size(rng, 256, 4096, 16), "tokens": int(_log(rng, 1, 65)), "enc": enc}
    if kind == "step":
        c = {"kind": kind, "tokens": int(_log(rng, 1, 257)), "mode": mode, "enc": enc, **_layer(rng)}
        c["layers"] = max(1, min(16, round(MAX_STEP_WEIGHTS / 2 / _layer_weights(c))))
        return c
    if kind == "prefill" or kind == "fp8act":
        c = {"kind": kind, "tokens": int(_log(rng, 257, 8193)), "enc": enc, **_layer(rng)}
        if kind == "prefill":
            c["mode"] = mode
        c["tokens"] = min(c["tokens"], int(MAX_FLOPS / 2 / _layer_weights(c)))
        return c
    if kind == "moe":
        experts = rng.choice([4, 8, 8, 16, 32, 64])
        hidden = _size(rng, 1024, 4096, 16)
        # expert feed-forward sizes shrink as their number grows; never more weights than the listed case has
        ffn = max(256, 16 * int(min(14336.0, 8 * 4096 * 14336 / (experts * hidden)) * rng.uniform(0.3, 1.0) / 16))
        return {"kind": kind, "tokens": int(_log(rng, 1, 2049)), "mode": mode, "experts": experts, "hidden": hidden, "ffn": ffn}
    return {"kind": "load", "outliers": rng.choice([0, 0, 1, 8]), **_layer(rng)}


def _linears(c):
    """(rows, columns) of the layer's four linears."""
    h, f = c["hidden"], c["ffn"]
    return [(c["qkv"], h), (h, h), (2 * f, h), (h, f)]


def _normal(shape, gen, std=1.0):
    return (torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32) * std).to(torch.float16)


def _planes(n, k, gen, enc, mode):
    p, r, _ = dps.dps_split_weights(_normal((n, k), gen, 0.02), enc)
    return p, (r if mode == dps.DPS_MODE_FULL else None)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    kind, s = case["kind"], {"kind": case["kind"]}
    if kind == "load":
        s["w"] = []
        for n, k in _linears(case):
            w = _normal((n, k), gen, 0.02)
            if case["outliers"]:
                at = torch.randint(0, n * k, (case["outliers"],), generator=gen, device="cuda")
                w.view(-1)[at] = (2.0 + 4.0 * torch.rand(case["outliers"], generator=gen, device="cuda")).to(torch.float16)
            s["w"].append(w)
        return s
    if kind == "moe":
        e, t, h, f = case["experts"], case["tokens"], case["hidden"], case["ffn"]
        s["mode"] = MODES[case["mode"]]
        s["enc"] = [dps.DPS_ENC_E4M3 if i % 4 != 3 else dps.DPS_ENC_E5M2 for i in range(e)]   # one layer in four out of range
        s["token"] = torch.arange(2 * t, device="cuda", dtype=torch.int32) // 2
        first = torch.randint(0, e, (t,), generator=gen, device="cuda")
        second = (first + 1 + torch.randint(0, e - 1, (t,), generator=gen, device="cuda")) % e
        s["expert"] = torch.stack([first, second], 1).reshape(-1).to(torch.int32)
        s["x"] = [_normal((t, h), gen), _normal((2 * t, f), gen)]
        s["planes"] = []
        for n, k in ((2 * f, h), (h, f)):
            p = torch.empty((e, n, k), dtype=torch.uint8, device="cuda")
            r = torch.empty_like(p)
            for i in range(e):
                dps.dps_split_weights(_normal((n, k), gen, 0.02), s["enc"][i], p[i], r[i])
            s["planes"].append((p, r if s["mode"] == dps.DPS_MODE_FULL else None))
        need = max(dps.dps_moe_workspace_bytes(2 * t, e, h), dps.dps_moe_workspace_bytes(2 * t, e, f))
        s["workspace"] = torch.empty(need, dtype=torch.uint8, device="cuda")
        return s
    s["enc"] = enc = ENCODINGS[case["enc"]]
    if kind == "single":
        s["x"] = _normal((case["tokens"], case["k"]), gen)
        s["p"], s["r"] = _planes(case["n"], case["k"], gen, enc, dps.DPS_MODE_FULL)
        return s
    s["mode"] = mode = dps.DPS_MODE_FAST if kind == "fp8act" else MODES[case["mode"]]
    m = case["tokens"]
    s["calls"] = [(_normal((m, k), gen), *_planes(n, k, gen, enc, mode)) for _ in range(case.get("layers", 1)) for n, k in _linears(case)]
    if kind == "step":
        s["y"] = [torch.empty((m, p.shape[0]), dtype=torch.float16, device="cuda") for _, p, _ in s["calls"]]

        def step():
            for (x, p, r), y in zip(s["calls"], s["y"]):
                dps.dps_linear(mode, enc, x, p, r, y)

        step()     # one-time set-up of the kernels stays out of the capture
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            step()
    return s


def run(state):
    kind = state["kind"]
    if kind == "step":
        state["graph"].replay()
        return state["y"]
    if kind == "single":
        return [dps.dps_linear(mode, state["enc"], state["x"], state["p"], state["r"]) for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL)]
    if kind == "prefill":
        return [dps.dps_linear(state["mode"], state["enc"], x, p, r) for x, p, r in state["calls"]]
    if kind == "fp8act":
        out = []
        for x, p, _ in state["calls"]:
            q, scale = dps.dps_quantize_activations(x)
            out.append((q, scale, dps.dps_linear_fp8act(state["enc"], q, scale, p)))
        return out
    if kind == "moe":
        (p1, r1), (p2, r2) = state["planes"]
        up = dps.dps_moe_linear(state["mode"], state["enc"], state["x"][0], state["token"], state["expert"], p1, r1,
                                workspace=state["workspace"])
        down = dps.dps_moe_linear(state["mode"], state["enc"], state["x"][1], None, state["expert"], p2, r2,
                                  workspace=state["workspace"])
        return up, down
    out = []
    for w in state["w"]:
        p, r, enc = dps.dps_split_weights(w)
        out.append((p, r, enc, dps.dps_reconstruct(p, r, enc)))
    return out


def work(case):
    kind = case["kind"]
    if kind == "load":      # split: FP16 in, two bytes out; reconstruction: two bytes in, FP16 out
        return {"bytes": 8.0 * _layer_weights(case), "flops": 0.0}
    if kind == "single":
        n, k, m = case["n"], case["k"], case["tokens"]
        return {"bytes": 3.0 * n * k + 2 * (2.0 * m * k + 2.0 * m * n), "flops": 4.0 * m * n * k}
    if kind == "moe":
        e, t, h, f = case["experts"], case["tokens"], case["hidden"], case["ffn"]
        hit = e * (1.0 - (1.0 - 2.0 / e) ** t)      # experts with at least one row, on average
        planes = 2.0 if case["mode"] == "full" else 1.0
        return {"bytes": hit * 3.0 * h * f * planes + 2.0 * t * h + 2 * t * (2.0 * 2 * f + 2.0 * f + 2.0 * h),
                "flops": 2.0 * 2 * t * 3.0 * h * f}
    m, layers = case["tokens"], case.get("layers", 1)
    planes = 2.0 if case.get("mode") == "full" else 1.0
    io = sum(2.0 * m * k + 2.0 * m * n for n, k in _linears(case))
    if kind == "fp8act":
        io += sum(2.0 * m * k + 8.0 * m for _, k in _linears(case))      # the codes and scales, written and read once
    return {"bytes": layers * (planes * _layer_weights(case) + io), "flops": layers * 2.0 * m * _layer_weights(case)}


def tolerance(case):
    if case["kind"] == "load":
        return "exact"
    # Products are exact in FP32, sums are FP32, the result is rounded once to FP16 (2^-11 relative at most).  Against the
    # same products summed in FP64 the cases show rel 2.1e-4 and max 5.1e-4; FP8 codes and scales are the same bit for bit.
    return {"rel": 8e-4, "max": 2e-3}


def _weights(w, enc, mode):
    """The weights a linear multiplies with, in FP64: all bits in full mode, those the persistent byte keeps in fast mode."""
    if mode == dps.DPS_MODE_FAST:
        keep = 7 if enc in (dps.DPS_ENC_E4M3, dps.DPS_ENC_E4M3_RN) else 8      # low bits of the word the byte leaves out
        half = 1 << (keep - 1) if enc in (dps.DPS_ENC_E4M3_RN, dps.DPS_ENC_E5M2_RN) else 0
        bits = (w.view(torch.int16).to(torch.int32) + half) >> keep << keep
        w = bits.to(torch.int16).view(torch.float16)
    return w.double()


def exact(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    kind = case["kind"]
    if kind == "load":      # bytes, the same in every implementation
        return None
    if kind == "moe":
        e, t, h, f = case["experts"], case["tokens"], case["hidden"], case["ffn"]
        mode = MODES[case["mode"]]
        first = torch.randint(0, e, (t,), generator=gen, device="cuda")
        second = (first + 1 + torch.randint(0, e - 1, (t,), generator=gen, device="cuda")) % e
        expert = torch.stack([first, second], 1).reshape(-1)
        x = [_normal((t, h), gen).double().repeat_interleave(2, 0), _normal((2 * t, f), gen).double()]
        out = []
        for i, (n, k) in enumerate(((2 * f, h), (h, f))):
            y = torch.empty((2 * t, n), dtype=torch.float64, device="cuda")
            for j in range(e):
                w = _weights(_normal((n, k), gen, 0.02), dps.DPS_ENC_E4M3 if j % 4 != 3 else dps.DPS_ENC_E5M2, mode)
                rows = (expert == j).nonzero().view(-1)
                y[rows] = x[i][rows] @ w.T
            out.append(y)
        return tuple(out)
    enc = ENCODINGS[case["enc"]]
    if kind == "single":
        x, w = _normal((case["tokens"], case["k"]), gen).double(), _normal((case["n"], case["k"]), gen, 0.02)
        return [x @ _weights(w, enc, mode).T for mode in (dps.DPS_MODE_FAST, dps.DPS_MODE_FULL)]
    out = []
    for _ in range(case.get("layers", 1)):
        for n, k in _linears(case):
            x, w = _normal((case["tokens"], k), gen), _normal((n, k), gen, 0.02)
            if kind != "fp8act":
                out.append(x.double() @ _weights(w, enc, MODES[case["mode"]]).T)
                continue
            # the codes and the scales are FP32 by definition; the product of the codes is what has a 64-bit value
            top = x.float().abs().amax(1)
            scale = torch.where(top > 0, top / torch.full_like(top, 448.0), torch.ones_like(top))      # (a scalar divisor is turned into a factor)
            codes = (x.float() / scale[:, None]).to(torch.float8_e4m3fn).double()
            out.append((None, None, scale.double()[:, None] * (codes @ _weights(w, enc, dps.DPS_MODE_FAST).T)))
    return out
