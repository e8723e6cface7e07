"""The work a user of okq has it do, as cases that can be timed and compared.

Every case is a dict of plain values; its "kind" names the part of a user's program it stands for:

  decode         one `decode_attention` call over all layers of a cache that is already full (a serving loop that
                 batches the layers, or one layer's call of a model)
  generate       a model's inner loop: for every new token and every layer one `append` and one `decode_attention`
                 (or one call of each over all layers), from the same prompt each pass; a pass is `steps` tokens
  prefill        a fresh prompt goes into the cache: `quantize_keys` and `quantize_values` layer by layer
  ladder_encode  keys and values quantised at 2, 3 or 4 bits into the canonical cache of the bit-width ladder
  ladder_decode  attention over such a cache
  turboquant     the baseline codec there and back: encode, then decode
  calibrate      offline calibration of one KV head: attention weights and moments of a few sequences, and the three
                 rotations from the moments that earlier sequences left

Shapes come from `paper_2609_11582_b200.workloads` (7B and 30B-A3B shapes, 350 or 500 tokens per two-second chunk).
"""
from __future__ import annotations

import torch

from paper_2609_11582_b200 import binding as B
from paper_2609_11582_b200 import workloads as WL

D, W = 128, 32
RAW_TOKEN_BYTES = 2 * D * 2          # one raw fp16 key and value


# ------------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: one layer, one sequence, one KV head with seven query heads, a two-second context
        {"name": "decode tiny", "kind": "decode", "layers": 1, "batch": 1, "q_heads": 7, "kv_heads": 1, "tokens": 2048,
         "meta": "fp16", "schedule": "window", "rotations": "layer"},
        # the benchmark's step: 28 layers of the 7B shape, eight sequences of 16k tokens, all layers in one call
        {"name": "decode step7b", "kind": "decode", "layers": 28, "batch": 8, "q_heads": 28, "kv_heads": 4,
         "tokens": 16384, "meta": "fp16", "schedule": "window", "rotations": "layer"},
        # the paper's own setting for captioning: MXFP4 metadata, keys packed every 128 tokens, values behind a 128-token
        # window, rotations calibrated per head; a context that is no multiple of anything
        {"name": "decode caption mxfp4", "kind": "decode", "layers": 28, "batch": 8, "q_heads": 28, "kv_heads": 4,
         "tokens": 12345, "meta": "mxfp4", "schedule": "caption", "rotations": "head"},
        # one long recording: batch 1 at 131072 tokens, the window axis split over the whole GPU
        {"name": "decode long7b", "kind": "decode", "layers": 28, "batch": 1, "q_heads": 28, "kv_heads": 4,
         "tokens": 131072, "meta": "fp16", "schedule": "window", "rotations": "layer"},
        # the largest: the 30B-A3B shape, 16 sequences of 32k tokens
        {"name": "decode step30b", "kind": "decode", "layers": 48, "batch": 16, "q_heads": 32, "kv_heads": 4,
         "tokens": 32768, "meta": "fp16", "schedule": "window", "rotations": "layer"},
        # a model generating: append and attention layer by layer, 32 tokens (so one of them packs a window)
        {"name": "generate 7b", "kind": "generate", "layers": 28, "batch": 4, "q_heads": 28, "kv_heads": 4,
         "tokens": 4096, "steps": 32, "per_layer": True, "meta": "fp16", "schedule": "window", "rotations": "head"},
        # a long audio-visual prompt: 32k tokens through the bulk quantisers, 28 layers
        {"name": "prefill 32k", "kind": "prefill", "layers": 28, "batch": 1, "q_heads": 28, "kv_heads": 4,
         "tokens": 32768, "bulk": True, "heads_inner": False, "meta": "fp16", "schedule": "window",
         "rotations": "layer"},
        # a short ragged prompt as the projections leave it (heads inside tokens), default value quantiser, MXFP4
        {"name": "prefill prompt", "kind": "prefill", "layers": 28, "batch": 1, "q_heads": 28, "kv_heads": 4,
         "tokens": 1357, "bulk": False, "heads_inner": True, "meta": "mxfp4", "schedule": "window",
         "rotations": "head"},
        # the bit-width ladder: K3V3 written, K4V4 read
        {"name": "ladder encode k3v3", "kind": "ladder_encode", "batch": 8, "q_heads": 28, "kv_heads": 4,
         "tokens": 8192, "bits": 3},
        {"name": "ladder decode k4v4", "kind": "ladder_decode", "batch": 64, "q_heads": 28, "kv_heads": 4,
         "tokens": 8192, "bits": 4},
        # the baseline codec on one layer's keys: 8 sequences x 4 heads x 16k tokens
        {"name": "turboquant k2", "kind": "turboquant", "vectors": 524288, "bits": 2},
        # one KV head of the calibration set
        {"name": "calibrate", "kind": "calibrate", "group": 7, "tokens": 8192, "sequences": 2},
    ]


MOST_TOKEN_HEADS = 48 * 16 * 4 * 32768        # decode: the largest listed case
MOST_GENERATE_TOKEN_HEADS = 28 * 4 * 4 * 4096
MOST_PREFILL_TOKEN_HEADS = 28 * 4 * 32768
MOST_LADDER_TOKEN_HEADS = 64 * 4 * 8192
MOST_VECTORS = 1 << 21


def _log(rng, lo, hi):
    """An integer of [lo, hi], uniform over its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def _heads(rng):
    kv, group = rng.choice([(1, 7), (2, 8), (4, 7), (4, 8), (4, 5), (8, 4), (8, 1)])
    return {"q_heads": kv * group, "kv_heads": kv}


def _format(rng):
    return {"meta": rng.choice(["fp16", "mxfp4"]), "schedule": rng.choice(["window", "caption"]),
            "rotations": rng.choice(["layer", "head"])}


def draw(rng):
    kind = rng.choice(["decode"] * 8 + ["generate"] * 3 + ["prefill"] * 4 +
                      ["ladder_encode", "ladder_decode", "turboquant", "calibrate"])
    if kind == "decode":
        c = {"kind": kind, "layers": rng.choice([1, 1, 28, 48, rng.randint(2, 48)]), "batch": _log(rng, 1, 16), **_heads(rng)}
        top = MOST_TOKEN_HEADS // (c["layers"] * c["batch"] * c["kv_heads"])
        return {**c, "tokens": _log(rng, 64, min(131072, top)), **_format(rng)}
    if kind == "generate":
        c = {"kind": kind, "layers": rng.randint(1, 28), "batch": _log(rng, 1, 8), **_heads(rng)}
        # the prompt ends on a packing boundary of both schedules, so that a pass leaves it as it found it
        top = MOST_GENERATE_TOKEN_HEADS // (c["layers"] * c["batch"] * c["kv_heads"] * 128)
        return {**c, "tokens": 128 * _log(rng, 1, min(64, top)), "steps": rng.choice([8, 32]), "per_layer": rng.random() < 0.7,
                **_format(rng)}
    if kind == "prefill":
        c = {"kind": kind, "layers": rng.randint(1, 28), "batch": _log(rng, 1, 8), **_heads(rng)}
        top = MOST_PREFILL_TOKEN_HEADS // (c["layers"] * c["batch"] * c["kv_heads"])
        return {**c, "tokens": _log(rng, 33, min(32768, top)), "bulk": rng.random() < 0.7,
                "heads_inner": rng.random() < 0.5, **_format(rng)}
    if kind in ("ladder_encode", "ladder_decode"):
        c = {"kind": kind, "batch": _log(rng, 1, 64), **_heads(rng)}
        top = MOST_LADDER_TOKEN_HEADS // (c["batch"] * c["kv_heads"] * W)
        return {**c, "tokens": W * _log(rng, 4, min(512, top)), "bits": rng.choice([2, 3, 4])}
    if kind == "turboquant":
        return {"kind": kind, "vectors": _log(rng, 1000, MOST_VECTORS), "bits": rng.choice([2, 3, 4])}
    return {"kind": kind, "group": rng.randint(1, 8), "tokens": _log(rng, 512, 8192), "sequences": rng.randint(1, 3)}


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * seed + 20260911)
    return g


def _modality(case):
    """uint8 [tokens]: text around two-second chunks of video and audio tokens."""
    w = WL.WORKLOADS["step30b" if case.get("q_heads") == 32 else "step7b"]
    return WL.modality_layout(w, case["tokens"]).cuda()


def _keys(g, lead, n):
    """fp16 [*lead, n, 128]: a random walk over time plus noise, four channels of 128 at ten times the size."""
    k = torch.randn(*lead, n, D, generator=g, device="cuda").mul_(0.05)
    k = k.cumsum_(dim=-2)
    k += torch.randn(*lead, 1, D, generator=g, device="cuda")
    k += torch.randn(*lead, n, D, generator=g, device="cuda")
    amp = torch.ones(*lead, D, device="cuda")
    amp.scatter_(-1, torch.rand(*lead, D, generator=g, device="cuda").topk(4, dim=-1).indices, 10.0)
    return k.mul_(amp.unsqueeze(-2)).half()


def _values(g, lead, n, mod):
    """fp16 [*lead, n, 128]: 16 directions of each modality's own plus noise."""
    frames = torch.randn(*lead, 3, 16, D, generator=g, device="cuda").mul_(D ** -0.5)
    coef = torch.randn(*lead, n, 16, generator=g, device="cuda")
    v = torch.randn(*lead, n, D, generator=g, device="cuda").mul_(0.1)
    for m in range(3):
        v += (coef * (mod == m).unsqueeze(-1)) @ frames[..., m, :, :]
    return v.half()


def _signs(g, layers):
    return torch.randint(0, 2, (layers, D), generator=g, device="cuda").float().mul_(2).sub_(1)


def _rotations(g, layers, n_r):
    """fp32 [layers, n_r, 3, 128, 128] orthogonal: three reflections in random directions of a signed Hadamard matrix."""
    had = torch.ones(1, 1, device="cuda", dtype=torch.float64)
    while had.shape[0] < D:
        had = torch.cat([torch.cat([had, had], 1), torch.cat([had, -had], 1)], 0)
    r = (had * D ** -0.5).expand(layers, n_r, 3, D, D)
    r = r * (torch.randint(0, 2, (layers, n_r, 3, 1, D), generator=g, device="cuda").double() * 2 - 1)
    for _ in range(3):
        u = torch.randn(layers, n_r, 3, D, 1, generator=g, device="cuda", dtype=torch.float64)
        u = u / u.norm(dim=-2, keepdim=True)
        r = r - 2 * u @ (u.transpose(-1, -2) @ r)
    return r.float().contiguous()


def _formats(case):
    return {"meta_format": B.META_MXFP4 if case["meta"] == "mxfp4" else B.META_FP16,
            "schedule": B.SCHEDULE_CAPTION if case["schedule"] == "caption" else B.SCHEDULE_WINDOW}


def _n_r(case):
    return case["kv_heads"] if case["rotations"] == "head" else 1


def _filled_cache(case, g, signs, R, room):
    """A cache of the case's shape holding its `tokens` tokens, filled through the quantisers."""
    L, Bn, H, n = case["layers"], case["batch"], case["kv_heads"], case["tokens"]
    cache = B.Cache(L, Bn, H, case["q_heads"], (n + room + W - 1) // W * W, **_formats(case))
    mod = _modality(case)
    mod_b = mod.expand(Bn, n).contiguous()
    for layer in range(L):
        B.quantize_keys(cache, layer, _keys(g, (Bn, H), n), signs[layer])
        B.quantize_values(cache, layer, _values(g, (Bn, H), n, mod), mod_b, R[layer], bulk=True)
    return cache


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"case": case, "kind": kind}
    if kind in ("decode", "generate"):
        L, Bn, H, Hq = case["layers"], case["batch"], case["kv_heads"], case["q_heads"]
        steps = case.get("steps", 0)
        s["signs"], s["R"] = _signs(g, L), _rotations(g, L, _n_r(case))
        s["n_R"] = _n_r(case)
        s["cache"] = cache = _filled_cache(case, g, s["signs"], s["R"], steps)
        per_call = 1 if case.get("per_layer") else L
        s["workspace"] = torch.empty(B.decode_workspace_bytes(cache, per_call), dtype=torch.uint8, device="cuda")
        s["q"] = torch.randn(max(1, steps), L, Bn, Hq, D, generator=g, device="cuda").half()
        s["out"] = torch.empty(max(1, steps), L, Bn, Hq, D, device="cuda")
        if kind == "generate":
            s["prompt_len"] = cache.seq_len.clone()
            s["k_new"] = torch.randn(steps, L, Bn, H, D, generator=g, device="cuda").half()
            s["v_new"] = torch.randn(steps, L, Bn, H, D, generator=g, device="cuda").mul_(0.3).half()
            s["text"] = torch.full((Bn,), WL.TEXT, dtype=torch.uint8, device="cuda")
    elif kind == "prefill":
        L, Bn, H, n = case["layers"], case["batch"], case["kv_heads"], case["tokens"]
        s["signs"], s["R"] = _signs(g, L), _rotations(g, L, _n_r(case))
        s["cache"] = B.Cache(L, Bn, H, case["q_heads"], (n + W - 1) // W * W, **_formats(case))
        mod = _modality(case)
        s["modality"] = mod.expand(Bn, n).contiguous()

        def layout(x):   # heads inside tokens: what a projection [batch, token, head * 128] gives
            return x.transpose(1, 2).contiguous().transpose(1, 2) if case["heads_inner"] else x
        s["k"] = [layout(_keys(g, (Bn, H), n)) for _ in range(L)]
        s["v"] = [layout(_values(g, (Bn, H), n, mod)) for _ in range(L)]
    elif kind in ("ladder_encode", "ladder_decode"):
        Bn, H, n = case["batch"], case["kv_heads"], case["tokens"]
        s["signs"], s["R"] = _signs(g, 1)[0], _rotations(g, 1, 1)[0]
        s["cache"] = cache = B.LadderCache(Bn, H, case["q_heads"], n, case["bits"])
        mod = _modality(case)
        s["modality"] = mod.expand(Bn, n).contiguous()
        s["k"], s["v"] = _keys(g, (Bn, H), n), _values(g, (Bn, H), n, mod)
        if kind == "ladder_decode":
            B.ladder_quantize_keys(cache, s.pop("k"), s["signs"])
            B.ladder_quantize_values(cache, s.pop("v"), s["modality"], s["R"])
            s["q"] = torch.randn(Bn, case["q_heads"], D, generator=g, device="cuda").half()
            s["out"] = torch.empty(Bn, case["q_heads"], D, device="cuda")
    elif kind == "turboquant":
        s["signs"] = _signs(g, 1)[0]
        s["x"] = _keys(g, (), case["vectors"])
    else:
        n, G = case["tokens"], case["group"]
        s["signs"] = _signs(g, 1)[0]
        mod = _modality(case)
        s["modality"] = mod
        s["workspace"] = B.calib_workspace(G, n)
        s["sequences"] = [(torch.randn(G, n, D, generator=g, device="cuda").half(), _keys(g, (), n), _values(g, (), n, mod))
                          for _ in range(case["sequences"])]
        # moments of the sequences that came before: a falling spectrum in a basis of each modality's own
        basis = _rotations(g, 1, 1)[0, 0].double()
        lam = torch.logspace(1, -2, D, device="cuda", dtype=torch.float64)
        lam = lam * (1 + 0.3 * torch.rand(3, D, generator=g, device="cuda", dtype=torch.float64))
        s["moments"] = list(((basis * lam[:, None, :]) @ basis.transpose(1, 2)).float().contiguous())
    return s


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "decode":
        B.decode_attention(s["cache"], 0, case["layers"], s["q"], s["signs"], s["R"], s["workspace"], s["out"], n_R=s["n_R"])
        return s["out"]
    if kind == "generate":
        cache, L = s["cache"], case["layers"]
        cache.seq_len.copy_(s["prompt_len"])
        for i in range(case["steps"]):
            k, v, q, out = s["k_new"][i], s["v_new"][i], s["q"][i], s["out"][i]
            if case["per_layer"]:
                for layer in range(L):
                    sg, R = s["signs"][layer], s["R"][layer]
                    B.append(cache, layer, 1, k[layer], v[layer], s["text"], sg, R, n_R=s["n_R"])
                    B.decode_attention(cache, layer, 1, q[layer], sg, R, s["workspace"], out[layer], n_R=s["n_R"])
            else:
                B.append(cache, 0, L, k, v, s["text"], s["signs"], s["R"], n_R=s["n_R"])
                B.decode_attention(cache, 0, L, q, s["signs"], s["R"], s["workspace"], out, n_R=s["n_R"])
        return {"out": s["out"], "records": cache.records, "k_tail": cache.k_tail, "v_tail": cache.v_tail,
                "modality": cache.modality, "seq_len": cache.seq_len, "status": cache.status}
    if kind == "prefill":
        cache = s["cache"]
        for layer in range(case["layers"]):
            B.quantize_keys(cache, layer, s["k"][layer], s["signs"][layer])
            B.quantize_values(cache, layer, s["v"][layer], s["modality"], s["R"][layer], bulk=case["bulk"])
        return {"records": cache.records, "k_tail": cache.k_tail, "v_tail": cache.v_tail, "modality": cache.modality,
                "seq_len": cache.seq_len, "status": cache.status}
    if kind == "ladder_encode":
        cache = s["cache"]
        B.ladder_quantize_keys(cache, s["k"], s["signs"])
        B.ladder_quantize_values(cache, s["v"], s["modality"], s["R"])
        return {"k_codes": cache.k_codes, "k_norm": cache.k_norm, "k_meta": cache.k_meta, "v_codes": cache.v_codes,
                "v_norm": cache.v_norm, "modality": cache.modality}
    if kind == "ladder_decode":
        B.ladder_decode_attention(s["cache"], case["tokens"], s["q"], s["signs"], s["R"], s["out"])
        return s["out"]
    if kind == "turboquant":
        codes, norms = B.turboquant_encode(s["x"], s["signs"], case["bits"])
        return codes, norms, B.turboquant_decode(codes, norms, s["signs"], case["bits"])
    outs = []
    for q, k, v in s["sequences"]:
        w = B.calib_attention_weights(q, k, s["workspace"])
        outs += [w, B.calib_moments(v, w, s["modality"], s["workspace"])]
    for C in s["moments"]:
        R, lam, _ = B.calib_rotation(C, s["signs"], s["workspace"])
        outs += [R, lam]
    return outs


# ------------------------------------------------------------------------------------------------ what it needs
def _packed(case, n):
    """(packed keys, packed values) of a sequence of n tokens."""
    if case["schedule"] == "caption":
        return n - n % 128, max(0, n - 128) // W * W
    return n - n % W, n - n % W


def _decode_work(case, n):
    """Bytes and operations of attention over n tokens for all layers, sequences and heads."""
    L, Bn, H, Hq = case["layers"], case["batch"], case["kv_heads"], case["q_heads"]
    units = L * Bn * H
    kp, vp = _packed(case, n)
    meta = 136 / W if case["meta"] == "mxfp4" else 512 / W
    cached = kp * (meta + 2 + 32) + vp * (2 + 32) + (n - kp) * 2 * D + (n - vp) * 2 * D
    rot = L * _n_r(case) * 3 * D * D * 4
    return units * cached + Bn * vp + rot + L * Bn * Hq * D * (2 + 4), L * Bn * Hq * (4.0 * D * n + 3 * 2 * D * D)


def work(case):
    kind = case["kind"]
    if kind == "decode":
        b, f = _decode_work(case, case["tokens"])
        return {"bytes": b, "flops": f}
    if kind == "generate":
        b = f = 0.0
        token = case["layers"] * case["batch"] * case["kv_heads"] * RAW_TOKEN_BYTES
        for i in range(case["steps"]):
            db, df = _decode_work(case, case["tokens"] + i + 1)
            b, f = b + db + 2 * token, f + df
        return {"bytes": b, "flops": f}
    if kind == "prefill":
        L, Bn, H, n = case["layers"], case["batch"], case["kv_heads"], case["tokens"]
        kp, vp = _packed(case, n)
        meta = 136 / W if case["meta"] == "mxfp4" else 512 / W
        unit = n * RAW_TOKEN_BYTES + kp * (meta + 34) + vp * 34 + (n - kp + n - vp) * 2 * D
        # rotation of the values, butterflies of the keys
        return {"bytes": L * (Bn * H * unit + _n_r(case) * 3 * D * D * 4), "flops": L * Bn * H * n * (2.0 * D * D + 7 * D)}
    if kind in ("ladder_encode", "ladder_decode"):
        units, n = case["batch"] * case["kv_heads"], case["tokens"]
        cached = units * n * (2 * 16 * case["bits"] + 4 + 512 / W) + case["batch"] * n
        if kind == "ladder_encode":
            return {"bytes": cached + units * n * RAW_TOKEN_BYTES, "flops": units * n * (2.0 * D * D + 7 * D)}
        return {"bytes": cached + case["batch"] * case["q_heads"] * D * 6, "flops": case["batch"] * case["q_heads"] * 4.0 * D * n}
    if kind == "turboquant":
        n = case["vectors"]
        row = 16 * case["bits"] + 2
        return {"bytes": n * (2 * D + 2 * row + 4 * D), "flops": n * 2 * 7.0 * D}
    n, G, S = case["tokens"], case["group"], case["sequences"]
    return {"bytes": S * (n * D * 2 * (G + 2) + 9 * n + 3 * D * D * 4) + 6 * D * D * 4,
            "flops": S * (G * n * n * float(D) + 2.0 * n * D * D) + 3 * 9.0 * D ** 3}


def tolerance(case):
    kind = case["kind"]
    if kind in ("prefill", "ladder_encode"):
        return "exact"                       # codes, norms and metadata are fixed bit for bit
    if kind in ("decode", "generate"):
        return {"rel": 1e-3}                 # fp16 softmax numerators (2^-11); packed bytes stay the same
    if kind == "calibrate":
        return {"rel": 1e-3}                 # fp16 products in the scores
    return {"rel": 1e-5}                     # fp32 arithmetic
