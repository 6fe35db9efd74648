"""The work that performance is measured on: calls of the public entry points
(``paper_2608_28003_gb300.binding``) at the sizes a Gemma-3-1B-shaped decoder (26 layers, hidden
1152, FFN 6912, 4 query heads on 1 key/value head of 256, vocabulary 262144) gives them, in the
three precisions of the library, from one token to a 2048-token prefill.

A case is a dict: ``op`` is the entry point (``linear``, ``ffn``, ``head``, ``decode``,
``prefill``), ``prec`` the precision (``w8a8``, ``bf16``, ``fp8``), the rest its sizes; decoder
cases carry the precision mask as layer bits.  Weights are N(0, 0.02) bf16, activations N(0, 1) bf16
with 1 % of the channels x20 (the regime SmoothQuant is made for; lm_head inputs are unit-RMS rows,
as after the final norm), calibration statistics the largest magnitudes over 512 calibration rows
with the same outlier channels.  Everything is drawn on the GPU from the seed alone.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as Fn

from paper_2608_28003_gb300 import binding as B

LAYERS, HIDDEN, INTER, VOCAB = 26, 1152, 6912, 262144
N_Q, N_KV, HEAD = 4, 1, 256
QKV, Q_DIM = (N_Q + 2 * N_KV) * HEAD, N_Q * HEAD
WINDOW, GLOBAL_LAYERS, EPS = 1024, (0, 6, 12, 18), 1e-6
CALIB_ROWS = 512
MASK_5_5 = B.GROUP_BITS["5+5"]


def listed():
    return [
        # one attention projection of one decode token: the smallest call, launch and latency only
        {"name": "linear_o_w8a8_m1", "op": "linear", "prec": "w8a8", "m": 1, "k": Q_DIM, "n": HIDDEN, "bias": False},
        # the single gate projection of a 16-sequence decode batch
        {"name": "linear_gate_w8a8_m16", "op": "linear", "prec": "w8a8", "m": 16, "k": HIDDEN, "n": INTER,
         "bias": False},
        # q/k/v of a layer left in bf16, a short prompt of an odd length, with a bias
        {"name": "linear_qkv_bf16_m37", "op": "linear", "prec": "bf16", "m": 37, "k": HIDDEN, "n": QKV, "bias": True},
        # the FFN block of a decode batch of 8, W8A8
        {"name": "ffn_w8a8_m8", "op": "ffn", "prec": "w8a8", "m": 8, "hidden": HIDDEN, "inter": INTER},
        # the FFN block of a large decode batch or a short prompt, W8A8
        {"name": "ffn_w8a8_m64", "op": "ffn", "prec": "w8a8", "m": 64, "hidden": HIDDEN, "inter": INTER},
        # the FFN block of a long prompt, W8A8
        {"name": "ffn_w8a8_m2048", "op": "ffn", "prec": "w8a8", "m": 2048, "hidden": HIDDEN, "inter": INTER},
        # the FFN block of a medium prompt in the FP8 variant
        {"name": "ffn_fp8_m512", "op": "ffn", "prec": "fp8", "m": 512, "hidden": HIDDEN, "inter": INTER},
        # lm_head of a decode batch of 16, W8A8: logits and top-1
        {"name": "head_w8a8_m16", "op": "head", "prec": "w8a8", "m": 16, "hidden": HIDDEN, "vocab": VOCAB},
        # lm_head over a teacher-forced stretch of an odd length left in bf16: logits and top-1
        {"name": "head_bf16_m509", "op": "head", "prec": "bf16", "m": 509, "hidden": HIDDEN, "vocab": VOCAB},
        # one decode token of one sequence under the paper's chosen mask (FFN 5+5 and lm_head in W8A8)
        {"name": "decode_b1", "op": "decode", "batch": 1, "pos": 160, "ffn": MASK_5_5, "attn": 0, "lm": 1},
        # one decode token of 8 sequences, the same mask
        {"name": "decode_b8", "op": "decode", "batch": 8, "pos": 160, "ffn": MASK_5_5, "attn": 0, "lm": 1},
        # a 2048-token prefill with every position's logits (the teacher-forced quality evaluation), bf16
        {"name": "prefill_t2048", "op": "prefill", "batch": 1, "t": 2048, "ffn": 0, "attn": 0, "lm": 0},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _log16(rng, lo, hi):
    return 16 * _log_int(rng, lo // 16, hi // 16)


def draw(rng):
    op = rng.choice(["linear", "linear", "linear", "linear", "ffn", "ffn", "ffn", "head", "head", "decode", "prefill"])
    if op == "linear":
        prec = rng.choice(["w8a8", "w8a8", "bf16", "fp8"])
        k, n = rng.choice([(HIDDEN, QKV), (Q_DIM, HIDDEN), (HIDDEN, INTER), (INTER, HIDDEN),
                           (_log16(rng, 256, 8192), _log16(rng, 256, 16384))])
        return {"op": op, "prec": prec, "m": _log_int(rng, 1, 2048), "k": k, "n": n, "bias": rng.random() < 0.5}
    if op == "ffn":
        prec = rng.choice(["w8a8", "w8a8", "bf16", "fp8"])
        h, f = rng.choice([(HIDDEN, INTER), (HIDDEN, INTER), (_log16(rng, 512, 2048), _log16(rng, 2048, 8192))])
        return {"op": op, "prec": prec, "m": _log_int(rng, 1, 2048), "hidden": h, "inter": f}
    if op == "head":
        return {"op": op, "prec": rng.choice(["w8a8", "bf16"]), "m": _log_int(rng, 1, 512), "hidden": HIDDEN,
                "vocab": VOCAB}
    ffn, attn, lm = rng.choice([(0, 0, 0), (0, 0, 1), (MASK_5_5, 0, 1)])
    if op == "decode":
        batch = _log_int(rng, 1, 32)
        return {"op": op, "batch": batch, "pos": _log_int(rng, 16, 2000 // batch), "ffn": ffn, "attn": attn, "lm": lm}
    return {"op": op, "batch": 1, "t": _log_int(rng, 12, 2000), "ffn": ffn, "attn": attn, "lm": lm}


# ------------------------------------------------------------------------------- inputs
def _gen(seed, *keys):
    g = torch.Generator(device="cuda")
    s = int(seed) & 0xFFFFFFFF
    for k in keys:
        s = (s * 1000003 + 7919 * (int(k) + 1)) & 0x7FFFFFFFFFFF
    g.manual_seed(s)
    return g


def _weight(n, k, g):
    return (torch.randn(n, k, device="cuda", generator=g, dtype=torch.bfloat16) * 0.02).contiguous()


def _acts(m, k, g, outliers):
    x = torch.randn(m, k, device="cuda", generator=g)
    x[:, outliers] *= 20.0
    return x.to(torch.bfloat16)


def _outliers(k, g):
    return torch.randperm(k, device="cuda", generator=g)[: max(1, round(0.01 * k))]


def _unit_rows(m, k, g):
    x = torch.randn(m, k, device="cuda", generator=g)
    return (x * torch.rsqrt(x.square().mean(dim=1, keepdim=True))).to(torch.bfloat16)


def _absmax(x):
    return x.float().abs().amax(dim=0)


def _linear_inputs(c, seed):
    g = _gen(seed, 1)
    ch = _outliers(c["k"], g)
    d = {"w": _weight(c["n"], c["k"], g), "x": _acts(c["m"], c["k"], g, ch),
         "stat": _absmax(_acts(CALIB_ROWS, c["k"], g, ch))}
    d["bias"] = torch.randn(c["n"], device="cuda", generator=g) if c["bias"] else None
    return d


def _ffn_inputs(c, seed):
    g = _gen(seed, 2)
    H, I = c["hidden"], c["inter"]
    ch = _outliers(H, g)
    d = {"wg": _weight(I, H, g), "wu": _weight(I, H, g), "wd": _weight(H, I, g), "x": _acts(c["m"], H, g, ch)}
    cal = _acts(CALIB_ROWS, H, g, ch)
    d["stat_x"] = _absmax(cal)
    h = Fn.gelu(cal.float() @ d["wg"].float().t(), approximate="tanh") * (cal.float() @ d["wu"].float().t())
    d["stat_h"] = _absmax(h.to(torch.bfloat16))
    return d


def _head_inputs(c, seed):
    g = _gen(seed, 3)
    return {"w": _weight(c["vocab"], c["hidden"], g), "x": _unit_rows(c["m"], c["hidden"], g),
            "stat": _absmax(_unit_rows(CALIB_ROWS, c["hidden"], g))}


def _decoder_inputs(c, seed):
    g = _gen(seed, 4)
    w = {"wqkv": [_weight(QKV, HIDDEN, g) for _ in range(LAYERS)],
         "wo": [_weight(HIDDEN, Q_DIM, g) for _ in range(LAYERS)],
         "wg": [_weight(INTER, HIDDEN, g) for _ in range(LAYERS)],
         "wu": [_weight(INTER, HIDDEN, g) for _ in range(LAYERS)],
         "wd": [_weight(HIDDEN, INTER, g) for _ in range(LAYERS)],
         "embed": _weight(VOCAB, HIDDEN, g)}

    def mult(n, lo, hi):
        return torch.empty(n, device="cuda").uniform_(lo, hi, generator=g)

    # pre-norm multipliers around 1; post-norm ones below it, as in a trained sandwich-norm decoder,
    # where each sublayer adds a fraction of the residual stream's size
    norms = {"ln_in": [mult(HIDDEN, 0.5, 1.5) for _ in range(LAYERS)],
             "ln_post_attn": [mult(HIDDEN, 0.03, 0.15) for _ in range(LAYERS)],
             "ln_pre_ffn": [mult(HIDDEN, 0.5, 1.5) for _ in range(LAYERS)],
             "ln_post_ffn": [mult(HIDDEN, 0.03, 0.15) for _ in range(LAYERS)],
             "q_norm": [mult(HEAD, 0.5, 1.5) for _ in range(LAYERS)],
             "k_norm": [mult(HEAD, 0.5, 1.5) for _ in range(LAYERS)],
             "final_norm": mult(HIDDEN, 0.5, 1.5)}
    # a saved calibration (per layer: q/k/v, o, gate/up and down inputs; then the lm_head input):
    # statistics of the sizes that the decoder's activations reach
    parts = []
    for l in range(LAYERS):
        parts += [4.5 * norms["ln_in"][l], mult(Q_DIM, 0.5, 2.0), 4.5 * norms["ln_pre_ffn"][l], mult(INTER, 0.5, 4.0)]
    stats = torch.cat(parts + [4.5 * norms["final_norm"]])
    batch = c["batch"]
    t = c["t"] if c["op"] == "prefill" else c["pos"] + 1
    tokens = torch.randint(0, VOCAB, (batch, t), device="cuda", generator=g, dtype=torch.int32)
    return {"w": w, "norms": norms, "stats": stats, "tokens": tokens}


# ------------------------------------------------------------------------------- a pass
def prepare(case, seed):
    op = case["op"]
    if op == "linear":
        d = _linear_inputs(case, seed)
        if case["prec"] == "w8a8":
            w = B.prepare_weights(d["w"], d["stat"], want_f16=True)
        elif case["prec"] == "fp8":
            w = B.fp8_prepare_weights(d["w"], d["stat"])
        else:
            w = d["w"]
        return {"op": op, "prec": case["prec"], "w": w, "x": d["x"], "bias": d["bias"]}
    if op == "ffn":
        d = _ffn_inputs(case, seed)
        H, I = case["hidden"], case["inter"]
        if case["prec"] == "w8a8":
            f = B.FfnWeights(H, I, gate_up=B.prepare_gate_up(d["wg"], d["wu"], d["stat_x"], want_f16=True),
                             down=B.prepare_weights(d["wd"], d["stat_h"], want_f16=True))
        elif case["prec"] == "fp8":
            f = B.Fp8FfnWeights(H, I, B.fp8_prepare_gate_up(d["wg"], d["wu"], d["stat_x"]),
                                B.fp8_prepare_weights(d["wd"], d["stat_h"]))
        else:
            f = B.FfnWeights(H, I, gate_up_bf16=B.interleave_gate_up(d["wg"], d["wu"]), down_bf16=d["wd"])
        return {"op": op, "prec": case["prec"], "f": f, "x": d["x"]}
    if op == "head":
        d = _head_inputs(case, seed)
        if case["prec"] == "w8a8":
            hd = B.HeadWeights(case["vocab"], case["hidden"], q=B.prepare_weights(d["w"], d["stat"], want_f16=True))
        else:
            hd = B.HeadWeights(case["vocab"], case["hidden"], bf16=d["w"])
        return {"op": op, "prec": case["prec"], "hd": hd, "x": d["x"]}
    d = _decoder_inputs(case, seed)
    batch, t = d["tokens"].shape
    cfg = B.DecoderConfig(max_batch=batch, max_seq=2048 + 64, max_tokens=max(128, batch * t))
    dec = B.Decoder(cfg, d["w"], d["norms"])
    if case["ffn"] or case["attn"] or case["lm"]:
        dec.set_stats(d["stats"].cpu().numpy())
        dec.prepare()
    dec.set_mask(case["ffn"], case["attn"], bool(case["lm"]))
    if op == "prefill":
        return {"op": op, "dec": dec, "tokens": d["tokens"]}
    pos = case["pos"]
    dec.forward(d["tokens"][:, :pos].contiguous(), 0, want_logits=False)
    return {"op": op, "dec": dec, "token": d["tokens"][:, pos].contiguous(), "pos": pos,
            "logits": torch.empty(batch, VOCAB, dtype=torch.float32, device="cuda")}


def run(state):
    op = state["op"]
    if op == "linear":
        if state["prec"] == "w8a8":
            return B.linear(state["w"], state["x"], bias=state["bias"])
        if state["prec"] == "fp8":
            return B.fp8_linear(state["w"], state["x"], bias=state["bias"])
        return B.linear_bf16(state["w"], state["x"], bias=state["bias"])
    if op == "ffn":
        if state["prec"] == "fp8":
            return B.fp8_ffn_block(state["f"], state["x"])
        return B.ffn_block(state["f"], B.W8A8_PREC_W8A8 if state["prec"] == "w8a8" else B.W8A8_PREC_BF16, state["x"])
    if op == "head":
        return B.lm_head(state["hd"], B.W8A8_PREC_W8A8 if state["prec"] == "w8a8" else B.W8A8_PREC_BF16, state["x"])
    # Decoder cases return the logits: the top-1 tokens are their argmax (held to it by the GPU
    # tests), and a random-init decoder's flat logits make them turn on the last bits.
    if op == "decode":
        return state["dec"].decode_step(state["token"], state["pos"], logits=state["logits"])[0]
    return state["dec"].forward(state["tokens"], 0, want_logits=True)[0]


# ---------------------------------------------------------------------------- the least work
def _linear_work(prec, m, n, k, out_bytes):
    wb = 2 if prec == "bf16" else 1
    scales = 0 if prec == "bf16" else 4 * (n + k)
    return n * k * wb + scales + 2 * m * k + out_bytes * m * n, 2 * m * n * k


def work(case):
    op = case["op"]
    if op == "linear":
        b, f = _linear_work(case["prec"], case["m"], case["n"], case["k"], 2)
        return {"bytes": b + (4 * case["n"] if case["bias"] else 0), "flops": f}
    if op == "ffn":
        b0, f0 = _linear_work(case["prec"], case["m"], 2 * case["inter"], case["hidden"], 0)
        b1, f1 = _linear_work(case["prec"], case["m"], case["hidden"], case["inter"], 2)
        return {"bytes": b0 + b1 - 2 * case["m"] * case["inter"], "flops": f0 + f1}
    if op == "head":
        b, f = _linear_work(case["prec"], case["m"], case["vocab"], case["hidden"], 4)
        return {"bytes": b + 4 * case["m"], "flops": f}
    batch = case["batch"]
    t, ctx = (case["t"], 0) if op == "prefill" else (1, case["pos"])
    m = batch * t
    nbytes, flops = 4 * m + 4 * m * VOCAB, 0
    for l in range(LAYERS):
        f8 = "w8a8" if (case["ffn"] >> l) & 1 else "bf16"
        a8 = "w8a8" if (case["attn"] >> l) & 1 else "bf16"
        for prec, n, k in ((a8, QKV, HIDDEN), (a8, HIDDEN, Q_DIM), (f8, 2 * INTER, HIDDEN), (f8, HIDDEN, INTER)):
            b, f = _linear_work(prec, 0, n, k, 0)
            nbytes += b
            flops += 2 * m * n * k
        span = ctx + t if l in GLOBAL_LAYERS else min(WINDOW, ctx + t)
        nbytes += 2 * batch * 2 * N_KV * HEAD * (min(ctx, span) + t)  # cached keys and values, read and new
        # attended (query, key) pairs
        pairs = sum(min(ctx + i + 1, span) for i in range(t))
        flops += 4 * batch * pairs * N_Q * HEAD
    b, f = _linear_work("w8a8" if case["lm"] else "bf16", 0, VOCAB, HIDDEN, 0)
    return {"bytes": nbytes + b, "flops": flops + 2 * m * VOCAB * HIDDEN}


def tolerance(case):
    if case["op"] in ("decode", "prefill"):
        return TOL_DECODER_INT8 if case["ffn"] or case["attn"] or case["lm"] else TOL_DECODER
    if case["prec"] == "w8a8":
        return "exact"  # integer sums and documented fp32 roundings: every output bit is defined
    if case["op"] == "head":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.005}  # fp32 sums in another order; top-1 ties
    if case["op"] == "ffn":
        return {"rel": 1e-2, "max": 1e-1}  # bf16 h and y, fp32 sums in another order
    return {"rel": 8e-3, "max": 4e-2}  # bf16 outputs of fp32 sums in another order


TOL_DECODER = {"rel": 0.02, "max": 0.2}
TOL_DECODER_INT8 = {"rel": 0.03, "max": 0.3}


# ---------------------------------------------------------------------------- 64-bit results
def _codes(v, qmax):
    """Symmetric codes of the rows of fp32 v: (codes as fp64, scales as fp64), the quantiser's
    definition: s = max / qmax, code = round(v * (qmax / max)), nearest even (e4m3 for 448)."""
    m = v.abs().amax(dim=1, keepdim=True)
    r = torch.where(m > 0, qmax / m, torch.zeros_like(m))
    if qmax == 127.0:
        q = torch.round(v * r).clamp_(-127, 127)
    else:
        q = (v * r).clamp_(-448, 448).to(torch.float8_e4m3fn).float()
    return q.double(), (m / qmax).double()


def _smoothing(ws, stat):
    aw = torch.stack([w.float().abs().amax(dim=0) for w in ws]).amax(dim=0)
    d = torch.sqrt(stat) / torch.sqrt(aw)
    return torch.where((stat == 0) | (aw == 0) | ~torch.isfinite(d) | (d == 0), torch.ones_like(d), d)


def _q_linear(x_bf16, ws, stat, qmax, chunk=16384):
    """x W^T of each matrix in ws (they share the smoothing) with quantised operands, exact sums."""
    d = _smoothing(ws, stat)
    xq, sx = _codes(x_bf16.float() * (1.0 / d), qmax)
    out = []
    for w in ws:
        y = torch.empty(x_bf16.shape[0], w.shape[0], dtype=torch.float64, device="cuda")
        for i in range(0, w.shape[0], chunk):
            wq, sw = _codes(w[i:i + chunk].float() * d, qmax)
            y[:, i:i + chunk] = (xq @ wq.t()) * sx * sw.t()
        out.append(y)
    return out


def _lin64(x, w, prec, stat, chunk=16384):
    if prec != "bf16":
        return _q_linear(x.to(torch.bfloat16), [w], stat, 127.0 if prec == "w8a8" else 448.0)[0]
    x = x.double()
    return torch.cat([x @ w[i:i + chunk].double().t() for i in range(0, w.shape[0], chunk)], dim=1)


def _ffn64(x, wg, wu, wd, prec, stat_x, stat_h):
    if prec == "bf16":
        g, u = x.double() @ wg.double().t(), x.double() @ wu.double().t()
    else:
        g, u = _q_linear(x.to(torch.bfloat16), [wg, wu], stat_x, 127.0 if prec == "w8a8" else 448.0)
    return _lin64(Fn.gelu(g, approximate="tanh") * u, wd, prec, stat_h)


def _norm64(x, w):
    return x * torch.rsqrt(x.square().mean(dim=-1, keepdim=True) + EPS) * w.double()


def _decoder64(case, d):
    tokens, w, n = d["tokens"].long(), d["w"], d["norms"]
    batch, t = tokens.shape
    r = w["embed"][tokens].double() * math.sqrt(HIDDEN)
    pos = torch.arange(t, device="cuda", dtype=torch.float64)
    half = torch.arange(HEAD // 2, device="cuda", dtype=torch.float64)
    gap = pos[:, None] - pos[None, :]
    stride, at = 2 * HIDDEN + Q_DIM + INTER, 0
    for l in range(LAYERS):
        at = l * stride
        s = d["stats"]
        s_qkv, s_o = s[at:at + HIDDEN], s[at + HIDDEN:at + HIDDEN + Q_DIM]
        s_gu = s[at + HIDDEN + Q_DIM:at + 2 * HIDDEN + Q_DIM]
        s_dn = s[at + 2 * HIDDEN + Q_DIM:at + stride]
        f8 = "w8a8" if (case["ffn"] >> l) & 1 else "bf16"
        a8 = "w8a8" if (case["attn"] >> l) & 1 else "bf16"
        glob = l in GLOBAL_LAYERS
        a = _norm64(r, n["ln_in"][l]).view(batch * t, HIDDEN)
        qkv = _lin64(a, w["wqkv"][l], a8, s_qkv).view(batch, t, N_Q + 2 * N_KV, HEAD)
        q, k, v = qkv[:, :, :N_Q], qkv[:, :, N_Q:N_Q + N_KV], qkv[:, :, N_Q + N_KV:]
        q, k = _norm64(q, n["q_norm"][l]), _norm64(k, n["k_norm"][l])
        ang = pos[:, None] * (1e6 if glob else 1e4) ** (-2.0 * half / HEAD)
        cos, sin = torch.cos(ang)[None, :, None, :], torch.sin(ang)[None, :, None, :]

        def rope(z):
            z1, z2 = z[..., :HEAD // 2], z[..., HEAD // 2:]
            return torch.cat([z1 * cos - z2 * sin, z2 * cos + z1 * sin], dim=-1)

        q, k = rope(q), rope(k)
        dead = (gap < 0) if glob else (gap < 0) | (gap >= WINDOW)
        o = torch.empty_like(q)
        for b in range(batch):
            for h in range(N_Q):
                kh = h * N_KV // N_Q
                sc = (q[b, :, h] @ k[b, :, kh].t()) / math.sqrt(HEAD)
                o[b, :, h] = torch.softmax(sc.masked_fill(dead, -math.inf), dim=-1) @ v[b, :, kh]
        y = _lin64(o.reshape(batch * t, Q_DIM), w["wo"][l], a8, s_o).view(batch, t, HIDDEN)
        r = r + _norm64(y, n["ln_post_attn"][l])
        a = _norm64(r, n["ln_pre_ffn"][l]).view(batch * t, HIDDEN)
        y = _ffn64(a, w["wg"][l], w["wu"][l], w["wd"][l], f8, s_gu, s_dn).view(batch, t, HIDDEN)
        r = r + _norm64(y, n["ln_post_ffn"][l])
    if case["op"] == "decode":
        r = r[:, -1:]
    a = _norm64(r, n["final_norm"]).reshape(-1, HIDDEN)
    return _lin64(a, w["embed"], "w8a8" if case["lm"] else "bf16", d["stats"][LAYERS * stride:])


def exact(case, seed):
    op = case["op"]
    if op == "linear":
        d = _linear_inputs(case, seed)
        y = _lin64(d["x"], d["w"], case["prec"], d["stat"])
        return y if d["bias"] is None else y + d["bias"].double()
    if op == "ffn":
        d = _ffn_inputs(case, seed)
        return _ffn64(d["x"], d["wg"], d["wu"], d["wd"], case["prec"], d["stat_x"], d["stat_h"])
    if op == "head":
        d = _head_inputs(case, seed)
        y = _lin64(d["x"], d["w"], case["prec"], d["stat"])
        return y, y.argmax(dim=1).to(torch.int32)
    return _decoder64(case, _decoder_inputs(case, seed))
