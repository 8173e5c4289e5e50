"""Performance cases of the framework's public entry points.

A case is one call (or one detect -> route/pack -> layer step) that a program
built on this package makes, with the sizes it makes it at: the batches of the
benchmark's workloads (a small fp32 model, one 8B-sized layer at batch 1, the
ragged batch of 16, the cached 32-layer stack's step, the video batch with
11.8k-row prefixes), plus sizes of the routing sweep and of the tests.

  listed()       the cases
  draw(rng)      one more case of the same ranges
  prepare(c, s)  the state a user's program holds before the call
  run(state)     one pass; returns its outputs
  work(c)        bytes and operations that one pass cannot do without
  tolerance(c)   how far a correct implementation of equal precision may be off
  exact(c, s)    the outputs in 64 bits, in plain torch

Lengths are texts: "3012x8" is eight sequences of 3012 rows, "70,33" two.
"""
import math
import random

import torch

from paper_2607_14557_gb300 import driver as D
from paper_2607_14557_gb300 import seer as S

EPS = 1e-5                                   # RMSNorm epsilon of every model here
TDT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
MODEL_8B = dict(d=4096, heads=32, ff=12288, dtype="bf16", act_eps=5e-3)
MAX_ROWS = 47000                             # rows of the largest drawn batch (the listed video batch has 47493)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest whole step: a tiny fp32 model, one sequence (launches and latency)
        dict(name="path_f32_b1", kind="path", dtype="f32", d=256, heads=4, ff=768, act_eps=3e-4, ctx="80", resp="41",
             window=128, rope=False),
        # fp32 validation of a small rotary model on a ragged batch
        dict(name="layer_f32_rope_b8", kind="layer", dtype="f32", d=512, heads=8, ff=1536, act_eps=3e-4,
             ctx="312,97,540,64,201,730,33,158", resp="41,17,77,103,9,60,25,128", pad="0,0,0,25,0,4,0,0", window=128,
             rope=True, hook=False),
        # interactive use: one image + question, one layer of an 8B model
        dict(MODEL_8B, name="path_8b_b1", kind="path", ctx="793", resp="49", window=256, rope=False),
        # throughput serving: the ragged batch of 16, detector to layer output
        dict(MODEL_8B, name="path_8b_ragged_b16", kind="path",
             ctx="2291,1572,805,1505,847,1513,2971,809,2985,3006,770,809,3005,3026,3037,2953",
             resp="368,184,106,307,204,17,40,356,113,191,247,353,183,144,312,98", window=1024, rope=False),
        # a rotary model's layer on a few short sequences; the step-0 hook counts near-zero activations
        dict(MODEL_8B, name="layer_8b_rope_hook_b4", kind="layer", ctx="615,161,1530,390", resp="256,256,256,256",
             pad="0,0,0,0", window=256, rope=True, hook=True),
        # video: 11.8k-row prefixes, attention dominates (the largest pass)
        dict(MODEL_8B, name="layer_8b_video_b4", kind="layer", ctx="11792x4", resp="41,37,106,141", pad="0,27,0,0",
             window=2048, rope=False, hook=False),
        # denoising steps with the prefix K/V cache: response rows only, 3012 cached rows each
        dict(MODEL_8B, name="cached_8b_b8", kind="cached", ctx="3012x8", resp="66,196,47,151,34,202,110,42"),
        # filling one layer's prefix cache for that batch
        dict(MODEL_8B, name="prefill_8b_b8", kind="prefill", ctx="3012x8", resp="66,196,47,151,34,202,110,42"),
        # the step-0 detector over the batch's full windows
        dict(MODEL_8B, name="detect_8b_b8", kind="detect", ctx="300x8", resp="66,196,47,151,34,202,110,42", window=512),
        # routing + compaction of a batch of 32 with odd lengths
        dict(MODEL_8B, name="pack_8b_b32", kind="pack", window=1024,
             ctx=",".join(str(729 * (1 + i % 5) + 32 + 3 * i) for i in range(32)),
             resp=",".join(str(17 + 37 * i % 384) for i in range(32))),
        # attention alone on bf16 q/k/v, odd ragged lengths, masked padding rows
        dict(name="attention_bf16_ragged", kind="attention", dtype="bf16", heads=32,
             lens="1437,333,129,2050,64,911,1,700", pad="0,25,0,3,0,11,0,0"),
        # the layer's f16 normalisation at an odd row count
        dict(name="norm_f16_rows", kind="norm", dtype="f16", d=4096, rows=9973),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _text(values):
    return ",".join(str(v) for v in values)


def draw(rng):
    kind = rng.choice(["path", "layer", "layer", "cached", "prefill", "detect", "pack", "attention", "norm"])
    if kind == "norm":
        return dict(kind="norm", dtype=rng.choice(["bf16", "f16"]), d=8 * _log(rng, 32, 512), rows=_log(rng, 1, MAX_ROWS))
    if kind == "attention":
        b, top = _log(rng, 1, 16), _log(rng, 16, 6000)
        lens = [_log(rng, max(1, top // 16), top) for _ in range(b)]
        pad = [rng.randint(0, (n - 1) // 4) if rng.random() < 0.3 else 0 for n in lens]
        return dict(kind="attention", dtype=rng.choice(["bf16", "f16", "f16"]), heads=rng.choice([2, 8, 32, 32]),
                    lens=_text(lens), pad=_text(pad))
    small = kind in ("path", "layer") and rng.random() < 0.25
    if small:
        hd = rng.choice([32, 64, 64, 128])
        heads = rng.choice([2, 4, 8]) if hd < 128 else rng.choice([2, 4])
        model = dict(dtype="f32", d=heads * hd, heads=heads, ff=4 * _log(rng, 64, 512), act_eps=3e-4)
    elif rng.random() < 0.6:
        model = dict(MODEL_8B)
    else:
        heads = rng.choice([2, 4, 8, 16])
        model = dict(dtype="bf16", d=128 * heads, heads=heads, ff=128 * _log(rng, heads, 6 * heads),
                     act_eps=3e-4 if heads <= 4 else 5e-3)
    b = _log(rng, 1, 16)
    window = _log(rng, 32, 256 if small else 1024)
    rows = 4000 if small else MAX_ROWS
    top = _log(rng, 16, max(16, min(12000, rows // b - window)))
    ctx = [_log(rng, max(1, top // 4), top) for _ in range(b)]
    resp = [min(window - 4, _log(rng, 8, window)) for _ in range(b)]
    case = dict(model, kind=kind, ctx=_text(ctx), resp=_text(resp))
    if kind in ("path", "layer"):
        case.update(window=window, rope=rng.random() < 0.3)
    if kind == "layer":
        case.update(hook=rng.random() < 0.3,
                    pad=_text(rng.randint(0, n) if rng.random() < 0.3 else 0 for n in resp))
    if kind in ("detect", "pack"):
        case.update(window=window)
    return case


# ------------------------------------------------------------------ sizes
def _list(text):
    out = []
    for part in text.split(","):
        n, _, times = part.partition("x")
        out += [int(n)] * int(times or 1)
    return out


def _cu(lens):
    cu = [0]
    for n in lens:
        cu.append(cu[-1] + n)
    return cu


def _packed(case):
    """(context, kept response rows, key counts) of each segment of a packed batch."""
    ctx, resp = _list(case["ctx"]), _list(case["resp"])
    pad = _list(case["pad"]) if "pad" in case else [0] * len(ctx)
    return ctx, [r + p for r, p in zip(resp, pad)], [c + r for c, r in zip(ctx, resp)]


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _i32(values):
    return torch.tensor(values, dtype=torch.int32, device="cuda")


def _model_weights(case, g, names=("w_qkv", "w_o", "w_gate", "w_up", "w_down", "g_attn", "g_mlp")):
    """Random-init weights N(0, 0.02^2) in the model's type, gains around 1."""
    d, ff, dt = case["d"], case["ff"], TDT[case["dtype"]]
    shapes = dict(w_qkv=(3 * d, d), w_o=(d, d), w_gate=(ff, d), w_up=(ff, d), w_down=(d, ff), g_attn=(d,), g_mlp=(d,))
    out = {}
    for name in names:
        r = _randn(g, *shapes[name])
        out[name] = (1.0 + 0.1 * r if name[0] == "g" else 0.02 * r).to(dt)
    return out


def _weights(case, g):
    model = _model_weights(case, g)
    run = model if case["dtype"] == "f32" else {k: D.f16_copy(v) for k, v in model.items()}
    return D.LayerWeights(model, run)


def _windows(case, g):
    """Full-window rows [context | window] of every sequence: N(0, 1), and past
    the end of the valid response the near-constant, near-zero suffix rows that
    the detector looks for."""
    ctx, resp, n, d = _list(case["ctx"]), _list(case["resp"]), case["window"], case["d"]
    cu = _cu([c + n for c in ctx])
    x = _randn(g, cu[-1], d)
    eos = 0.1 * _randn(g, d)
    for i, c in enumerate(ctx):
        a, b = cu[i] + c + resp[i] - 1, cu[i + 1]           # L* keeps one suffix row
        x[a:b] = eos + 0.05 * x[a:b]
    return x.to(TDT[case["dtype"]]), cu, [cu[i] + c for i, c in enumerate(ctx)]


def _dims(case):
    return S.make_dims(case["d"], case["heads"], case["d"] // case["heads"], case["ff"], EPS,
                       10000.0 if case.get("rope") else 0.0)


def prepare(case, seed):
    g = _generator(seed)
    st = {"case": case}
    kind = case["kind"]
    if kind == "norm":
        dt = TDT[case["dtype"]]
        st["x"] = _randn(g, case["rows"], case["d"]).to(dt)
        st["g"] = (1.0 + 0.1 * _randn(g, case["d"])).to(torch.float16)
        st["y"] = torch.empty((case["rows"], case["d"]), dtype=torch.float16, device="cuda")
        return st
    if kind == "attention":
        lens, pad = _list(case["lens"]), _list(case["pad"])
        heads, t = case["heads"], sum(lens)
        st["qkv"] = _randn(g, t, 3 * 128 * heads).to(TDT[case["dtype"]])
        st["o"] = torch.empty((t, 128 * heads), dtype=st["qkv"].dtype, device="cuda")
        st["cu"], st["kv"], st["t"], st["b"] = _i32(_cu(lens)), _i32([n - p for n, p in zip(lens, pad)]), t, len(lens)
        st["ws_bytes"] = S.seer_layer_workspace_size(S.make_dims(128 * heads, heads, 128, 128), case["dtype"], t, len(lens))
        st["ws"] = torch.empty(st["ws_bytes"], dtype=torch.uint8, device="cuda")
        return st
    dims, dtype, d = _dims(case), case["dtype"], case["d"]
    ctx, kept, keys = _packed(case)
    b = st["b"] = len(ctx)
    if kind in ("path", "detect", "pack"):
        n = case["window"]
        x, cu, first = _windows(case, g)
        if kind == "detect":
            w = D.LayerWeights(_model_weights(case, g, ("w_gate", "w_up")), {})
        elif kind == "path":
            w = _weights(case, g)
        else:
            w = None
        st.update(x=x, cu=_i32(cu), first=_i32(first), ctx=_i32(ctx), w=w)
        st["path"] = p = D.SeerPath(dims, dtype, b, n, cu[-1], S.make_params(case["act_eps"]))
        p.y.zero_()
        if kind == "pack":
            p.L_star.copy_(_i32(_list(case["resp"])))
        return st
    st.update(dims=dims, w=_weights(case, g), ctx=_i32(ctx))
    lens = [c + k for c, k in zip(ctx, kept)]
    cu = _cu(lens)
    st["t"], st["cu"], st["kv"] = cu[-1], _i32(cu), _i32(keys)
    if kind in ("layer", "prefill"):
        t = cu[-1]
        st["x"] = _randn(g, t, d).to(TDT[dtype])
    else:
        t = sum(kept)
        st["x"] = _randn(g, t, d).to(TDT[dtype])
        st["cu_resp"] = _i32(_cu(kept))
    st["rows"] = t
    st["ws_bytes"] = S.seer_layer_workspace_size(dims, dtype, t, b)
    st["ws"] = torch.empty(st["ws_bytes"], dtype=torch.uint8, device="cuda")
    inner = torch.float32 if dtype == "f32" else torch.float16
    if kind == "cached":
        st["cache"] = _randn(g, cu[-1], 2 * d).to(inner)
    if kind == "prefill":
        st["cache"] = torch.zeros((cu[-1], 2 * d), dtype=inner, device="cuda")
    else:
        st["y"] = torch.empty_like(st["x"])
    if kind == "layer":
        st["first"] = _i32([a + c for a, c in zip(cu, ctx)]) if case["hook"] else None
        st["counts"] = torch.empty(b * case["window"], dtype=torch.int32, device="cuda") if case["hook"] else None
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "path":
        p = st["path"]
        p.step(st["x"], st["cu"], st["first"], st["ctx"], st["w"])
        return {"counts": p.counts, "L": p.L_star, "i": p.i_star, "cu": p.cu, "kv": p.kv, "x": p.x_packed, "y": p.y}
    if kind == "detect":
        p = st["path"]
        p.detect(st["x"], st["first"], st["w"])
        return {"counts": p.counts, "L": p.L_star, "i": p.i_star}
    if kind == "pack":
        p = st["path"]
        p.pack(st["x"], st["cu"], st["ctx"])
        return {"x": p.x_packed, "cu": p.cu, "kv": p.kv, "meta": p.meta[1:]}      # word 0 numbers the calls
    if kind == "layer":
        hook = case["hook"]
        S.seer_layer_forward(st["w"].struct(), st["dims"], case["dtype"], st["x"], st["y"], st["cu"], st["kv"], st["b"],
                             st["t"], st["first"], case["window"] if hook else 0, case["act_eps"] if hook else 0.0,
                             st["counts"], st["ws"], st["ws_bytes"])
        return {"y": st["y"], "counts": st["counts"]} if hook else {"y": st["y"]}
    if kind == "cached":
        S.seer_layer_forward_cached(st["w"].struct(), st["dims"], case["dtype"], st["x"], st["y"], st["cu_resp"],
                                    st["ctx"], st["b"], st["rows"], st["cache"], st["cu"], st["kv"], st["t"], st["ws"],
                                    st["ws_bytes"])
        return {"y": st["y"], "cache": st["cache"]}
    if kind == "prefill":
        S.seer_kv_prefill(st["w"].struct(), st["dims"], case["dtype"], st["x"], st["cu"], st["ctx"], st["b"], st["rows"],
                          st["cache"], st["cu"], st["t"], st["ws"], st["ws_bytes"])
        return {"cache": st["cache"]}
    if kind == "attention":
        S.seer_attention(st["qkv"], st["o"], case["dtype"], st["cu"], st["kv"], st["b"], st["t"], case["heads"], 128,
                         st["ws"], st["ws_bytes"])
        return {"o": st["o"]}
    S.seer_rmsnorm(st["x"], case["dtype"], st["g"], st["y"], "f16", case["rows"], None, case["d"], EPS)
    return {"y": st["y"]}


# ------------------------------------------------------------------ the work of one pass
def work(case):
    kind = case["kind"]
    if kind == "norm":
        n = case["rows"] * case["d"]
        return {"bytes": 4 * n + 2 * case["d"], "flops": 4 * n}
    if kind == "attention":
        lens, pad, dm = _list(case["lens"]), _list(case["pad"]), 128 * case["heads"]
        return {"bytes": 2 * 4 * sum(lens) * dm, "flops": 4 * dm * sum(n * (n - p) for n, p in zip(lens, pad))}
    d, ff, es = case["d"], case["ff"], 4 if case["dtype"] == "f32" else 2
    ctx, kept, keys = _packed(case)
    rows = sum(ctx) + sum(kept)
    weights = es * (4 * d * d + 3 * d * ff + 2 * d)
    if kind == "detect":
        m = len(ctx) * case["window"]
        return {"bytes": es * (m * d + 2 * d * ff) + 4 * m, "flops": 4 * m * d * ff}
    if kind == "pack":
        return {"bytes": 2 * es * rows * d, "flops": 0}
    if kind == "prefill":
        m = sum(ctx)
        return {"bytes": es * (m * d + 2 * d * d + d + 2 * m * d), "flops": 4 * m * d * d}
    if kind == "cached":
        m = sum(kept)
        att = 4 * d * sum(k * n for k, n in zip(kept, keys))
        return {"bytes": es * (2 * m * d + 2 * rows * d) + weights, "flops": m * (8 * d * d + 6 * d * ff) + att}
    att = 4 * d * sum((c + k) * n for c, k, n in zip(ctx, kept, keys))
    layer = {"bytes": 2 * es * rows * d + weights, "flops": rows * (8 * d * d + 6 * d * ff) + att}
    if kind == "layer":
        return layer
    m = len(ctx) * case["window"]
    # the detector reads the model's own gate and up weights, a bf16 layer their f16 copies
    more = 2 * es * d * ff if es == 2 else 0
    return {"bytes": layer["bytes"] + more + es * m * d + 4 * m, "flops": layer["flops"] + 4 * m * d * ff}


def tolerance(case):
    # about four times the distances to exact() measured on a GB300: fp32 layers 4e-8 to 9e-8, 16-bit layers 1.7e-3
    # (their bf16 outputs), attention 2.3e-3 in bf16 and 4e-4 in f16, K/V projections and norms 2e-4 to 3e-4
    kind, f32 = case["kind"], case["dtype"] == "f32"
    if kind == "pack":
        return "exact"
    if kind == "detect":
        # whole numbers; a count moves by one where an activation lies within a rounding of the threshold
        return {"rel": 1e-3, "max": 0.05, "differ": 0.01}
    if f32:
        return {"rel": 1e-6, "max": 1e-4, "differ": 0.01}
    if kind == "norm":
        return {"rel": 1e-3, "max": 0.01}
    if kind == "attention":
        return {"rel": 9e-3 if case["dtype"] == "bf16" else 1.5e-3, "max": 0.1}
    if kind == "prefill":
        return {"rel": 1.2e-3, "max": 0.02}
    return {"rel": 7e-3, "max": 0.05, "differ": 0.01}


# ------------------------------------------------------------------ in 64 bits
def _f64(t):
    return t.to(torch.float64)


def _exact_norm(x, gain):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + EPS) * gain


def _exact_attention(q, k, v, heads):
    dh = q.shape[1] // heads
    split = lambda t: t.view(t.shape[0], heads, dh).transpose(0, 1)
    out = []
    for a, b, c in zip(split(q), split(k), split(v)):
        s = a @ b.T
        out.append(torch.softmax(s.mul_(1.0 / math.sqrt(dh)), dim=-1) @ c)
    return torch.cat(out, dim=1)


def _exact_rope(t, heads):
    """Pairs (i, i + dh/2) of each head turn by position * 10000^(-2i/dh)."""
    rows, d = t.shape
    half = d // heads // 2
    freq = 10000.0 ** (-torch.arange(half, dtype=torch.float64, device=t.device) / half)
    ang = torch.arange(rows, dtype=torch.float64, device=t.device)[:, None] * freq
    a, b = t.view(rows, heads, 2, half).unbind(2)
    c, s = ang.cos()[:, None], ang.sin()[:, None]
    return torch.stack((a * c - b * s, b * c + a * s), dim=2).reshape(rows, d)


def _exact_gates(x, w):
    return torch.nn.functional.silu(x @ _f64(w["w_gate"]).T) * (x @ _f64(w["w_up"]).T)


def _exact_mlp(h, w):
    """(output, activations) of the second half of the block."""
    act = _exact_gates(_exact_norm(h, _f64(w["g_mlp"])), w)
    return h + act @ _f64(w["w_down"]).T, act


def _exact_layer(x, w, heads, cu, keys, rope):
    d = x.shape[1]
    q, k, v = (_exact_norm(x, _f64(w["g_attn"])) @ _f64(w["w_qkv"]).T).split(d, dim=1)
    o = torch.empty_like(q)
    for a, b, n in zip(cu, cu[1:], keys):
        qq, kk = (_exact_rope(q[a:b], heads), _exact_rope(k[a:b], heads)) if rope else (q[a:b], k[a:b])
        o[a:b] = _exact_attention(qq, kk[:n], v[a:a + n], heads)
    del q, k, v
    return _exact_mlp(x + o @ _f64(w["w_o"]).T, w)


def _exact_boundaries(counts, ff):
    """Sec. 3.3 with its default thresholds: (L*, i*) of each row of counts."""
    n = counts.shape[1]
    ls, found = [], []
    for row in counts.tolist():
        s = [c / ff for c in row]
        hit = -1
        for i in range(1, n - 3 + 1):
            lo, hi = min(s[i:i + 3]), max(s[i:i + 3])
            if lo - s[i - 1] >= 0.03 and hi - lo <= 0.6 * (lo - s[i - 1]):
                hit = i
                break
        ls.append(hit + 1 if hit >= 0 else n)
        found.append(hit)
    return ls, found


def exact(case, seed):
    kind = case["kind"]
    if kind == "pack" or work(case)["flops"] > 5e12 or (kind == "path" and work(case)["flops"] > 2e12):
        return None                          # bytes only, or too long in 64 bits
    st = prepare(case, seed)
    if kind == "norm":
        return {"y": _exact_norm(_f64(st["x"]), _f64(st["g"]))}
    if kind == "attention":
        lens, pad, dm = _list(case["lens"]), _list(case["pad"]), 128 * case["heads"]
        cu, o = _cu(lens), torch.empty(st["o"].shape, dtype=torch.float64, device="cuda")
        for a, n, p in zip(cu, lens, pad):
            q, k, v = _f64(st["qkv"][a:a + n]).split(dm, dim=1)
            o[a:a + n] = _exact_attention(q, k[:n - p], v[:n - p], case["heads"])
        return {"o": o}
    ctx, kept, keys = _packed(case)
    d, ff, heads = case["d"], case["ff"], case["heads"]
    if kind == "detect" or kind == "path":
        n, first = case["window"], st["first"].tolist()
        m = st["w"].model
        win = torch.cat([_f64(st["x"][a:a + n]) for a in first])
        counts = (_exact_gates(win, m).abs_() < torch.tensor(case["act_eps"], dtype=torch.float32).item()).sum(1)
        ls, hits = _exact_boundaries(counts.view(len(ctx), n), ff)
        out = {"counts": counts.to(torch.int32), "L": _i32(ls), "i": _i32(hits)}
        if kind == "detect":
            return out
        return dict(out, cu=None, kv=None, x=None, y=_exact_path_layer(st, case, ls))
    w = st["w"].run
    x = _f64(st["x"])
    if kind == "prefill":
        cache = torch.zeros(st["cache"].shape, dtype=torch.float64, device="cuda")
        for a, c in zip(_cu([c + k for c, k in zip(ctx, kept)]), ctx):
            cache[a:a + c] = _exact_norm(x[a:a + c], _f64(w["g_attn"])) @ _f64(w["w_qkv"][d:]).T
        return {"cache": cache}
    if kind == "cached":
        cache = _f64(st["cache"])
        cu, cr = _cu([c + k for c, k in zip(ctx, kept)]), _cu(kept)
        qkv = _exact_norm(x, _f64(w["g_attn"])) @ _f64(w["w_qkv"]).T
        o = torch.empty_like(x)
        for i, c in enumerate(ctx):
            rows = slice(cr[i], cr[i + 1])
            cache[cu[i] + c:cu[i + 1]] = qkv[rows, d:]
            kv = cache[cu[i]:cu[i] + keys[i]]
            o[rows] = _exact_attention(qkv[rows, :d], kv[:, :d], kv[:, d:], heads)
        return {"y": _exact_mlp(x + o @ _f64(w["w_o"]).T, w)[0], "cache": cache}
    y, act = _exact_layer(x, w, heads, st["cu"].tolist(), keys, case["rope"])
    if not case["hook"]:
        return {"y": y}
    n, counts = case["window"], torch.zeros((len(ctx), case["window"]), dtype=torch.int32, device="cuda")
    zero = (act.abs_() < torch.tensor(case["act_eps"], dtype=torch.float32).item()).sum(1, dtype=torch.int32)
    for i, (a, k) in enumerate(zip(st["first"].tolist(), kept)):
        counts[i, :min(k, n)] = zero[a:a + min(k, n)]
    return {"y": y, "counts": counts.view(-1)}


def _exact_path_layer(st, case, ls):
    """The layer over the compacted rows: the buckets are the powers of two from
    8 below the window, and the window; a bucket's sequences are padded to it
    when it is over 4, has more than one and wastes at most a fifth (Sec. 3.4)."""
    n, ctx, cu = case["window"], _list(case["ctx"]), st["cu"].tolist()
    sizes = [8 << i for i in range(32) if 8 << i < n] + [n]
    bucket = [next(s for s in sizes if s >= l) for l in ls]
    kept = []
    for l, s in zip(ls, bucket):
        group = [v for v, t in zip(ls, bucket) if t == s]
        static = s > 4 and len(group) > 1 and 1.0 - sum(group) / (len(group) * s) <= 0.2
        kept.append(s if static else l)
    x = torch.cat([_f64(st["x"][a:a + c + k]) for a, c, k in zip(cu, ctx, kept)])
    y = torch.zeros(st["path"].y.shape, dtype=torch.float64, device="cuda")
    packed = _cu([c + k for c, k in zip(ctx, kept)])
    y[:packed[-1]] = _exact_layer(x, st["w"].run, case["heads"], packed, [c + l for c, l in zip(ctx, ls)], case["rope"])[0]
    return y


if __name__ == "__main__":
    for c in listed() + [dict(draw(random.Random(s)), name=f"drawn {s}") for s in range(8)]:
        print(c["name"], {k: v for k, v in c.items() if k != "name"}, work(c))
