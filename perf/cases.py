"""Workloads for timing the library through its public entry points.

Every case is one call (or one short loop of calls) that a serving or profiling
program makes: the compression of a prompt's KV cache right after its prefill
(one layer, a whole stack, or fused with the window rows' attention), the
selection from votes made elsewhere, decode steps over the ragged compressed
caches (all layers in one launch, or layer by layer in a captured graph), and
the two passes of the offline sensitivity profile. Shapes are those of the
repository's synthetic workloads and tests; `draw` spreads over their ranges.

Inputs follow the repository's synthetic recipe: keys N(0, 1) with a
per-channel lognormal(0, 0.5) scale and four sink tokens, values N(0, 1).
Window queries are N(0, 1) with a gain of 2, which gives attention as peaked as
a trained model's (logits of standard deviation about 2.5), so that votes span
orders of magnitude and few tokens tie at a selection threshold.

Kept cache rows are byte copies of input rows, so they are returned as the
integers behind their bits: `differ` is then the share of places that hold
another row, which is what a near-tie at the threshold resolved the other way
shows up as.
"""
from __future__ import annotations

import math

import torch

from paper_2608_08684_gb300 import ripple as R
from paper_2608_08684_gb300.serving import LayerDecodeLoop

DEV = "cuda"
_DT = {"bf16": torch.bfloat16, "f32": torch.float32}
_INT = {"bf16": torch.int16, "f32": torch.int32}


def listed():
    return [
        # the smallest prompt: four fp32 layers of 512 tokens, where launches count
        dict(name="layers_tiny_f32", kind="layers", layers=4, batch=1, q_heads=4, kv_heads=2,
             dim=64, seq=512, window=32, pool="max", pool_kernel=7, dtype="f32", budget=128,
             ratio=4.0),
        # one layer right after its prefill, votes wanted for inspection (8B shape, 8k prompt)
        dict(name="layer_8k", kind="layer", layers=1, batch=1, q_heads=32, kv_heads=8, dim=128,
             seq=8192, window=32, pool="max", pool_kernel=7, dtype="bf16", budget=512,
             ratio=1.0),
        # the headline workload: a batch of four 32k prompts, all 32 layers
        dict(name="layers_32k", kind="layers", layers=32, batch=4, q_heads=32, kv_heads=8,
             dim=128, seq=32768, window=32, pool="max", pool_kernel=7, dtype="bf16",
             budget=1024, ratio=8.0),
        # small heads, a 16-query window, average pooling and a ragged prompt length
        dict(name="layers_d64_avg", kind="layers", layers=16, batch=2, q_heads=32, kv_heads=8,
             dim=64, seq=6007, window=16, pool="avg", pool_kernel=5, dtype="bf16", budget=512,
             ratio=4.0),
        # eight query heads per KV head and a 128k prompt (16 layers of a 70B-shaped stack)
        dict(name="layers_128k_g8", kind="layers", layers=16, batch=1, q_heads=64, kv_heads=8,
             dim=128, seq=131072, window=32, pool="max", pool_kernel=7, dtype="bf16",
             budget=2048, ratio=8.0),
        # compression that also gives the window rows' attention output
        dict(name="layers_attn_32k", kind="attn", layers=8, batch=1, q_heads=32, kv_heads=8,
             dim=128, seq=32768, window=32, pool="max", pool_kernel=7, dtype="bf16",
             budget=1024, ratio=8.0),
        # votes made by another scorer: pooling, selection and gather of one layer
        dict(name="select_32k", kind="select", layers=1, batch=4, q_heads=32, kv_heads=8,
             dim=128, seq=32768, window=32, pool="max", pool_kernel=7, dtype="bf16",
             budget=1024, ratio=1.0),
        # a token of the serving loop: 32 single-layer steps replayed from a graph
        dict(name="serve_token", kind="loop", layers=32, batch=4, q_heads=32, kv_heads=8,
             dim=128, dtype="bf16", budget=1024, ratio=8.0, steps=1),
        # decode steps of the 32k workload, all layers in one launch
        dict(name="decode_32k", kind="decode", layers=32, batch=4, q_heads=32, kv_heads=8,
             dim=128, dtype="bf16", budget=1024, ratio=8.0, steps=8),
        # decode steps of the 70B shape
        dict(name="decode_128k_g8", kind="decode", layers=80, batch=1, q_heads=64, kv_heads=8,
             dim=128, dtype="bf16", budget=2048, ratio=8.0, steps=8),
        # profiling: the perturbed value cache of one layer (Eq. 6)
        dict(name="perturb_32k", kind="perturb", batch=4, kv_heads=8, dim=128, seq=32768,
             window=32, dtype="bf16"),
        # profiling: 32 perturbed runs against the reference over a 128k vocabulary (Eq. 7)
        dict(name="kl_32x32", kind="kl", sets=32, pos=32, vocab=128256, dtype="f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# shapes (query heads, KV heads, head dim, window, dtype) a compression call may have, in use:
# the 8B, 70B and small-head shapes, other windows, and fp32 caches
_SHAPES = [(32, 8, 128, 32, "bf16"), (32, 8, 128, 32, "bf16"), (64, 8, 128, 32, "bf16"),
           (32, 8, 128, 16, "bf16"), (32, 8, 64, 32, "bf16"), (8, 8, 128, 32, "bf16"),
           (24, 8, 128, 32, "bf16"), (16, 8, 128, 64, "bf16"), (4, 2, 64, 32, "f32"),
           (32, 8, 128, 32, "f32")]


def draw(rng):
    kind = rng.choice(["layers", "layers", "layer", "attn", "select", "loop", "decode", "decode",
                       "perturb", "kl"])
    if kind == "kl":
        c = dict(kind=kind, sets=rng.choice([1, 8, 16, 32]), pos=rng.choice([8, 16, 32]),
                 vocab=8 * _log(rng, 1000, 16032), dtype=rng.choice(["f32", "bf16"]))
        return c
    if kind == "perturb":
        return dict(kind=kind, batch=rng.choice([1, 2, 4]), kv_heads=rng.choice([2, 8]),
                    dim=rng.choice([64, 128]), seq=_log(rng, 512, 32768), window=32,
                    dtype=rng.choice(["bf16", "bf16", "f32"]))
    if kind in ("loop", "decode"):
        hq, hkv = rng.choice([(32, 8), (32, 8), (64, 8), (8, 8), (16, 8)])
        dim, dtype = rng.choice([(128, "bf16"), (128, "bf16"), (64, "bf16"), (64, "f32")])
        layers, batch = rng.choice([1, 4, 16, 32]), rng.choice([1, 2, 4, 8])
        steps = 1 if kind == "loop" else 8
        # at most 5 GB of cache rows read, as the largest listed steps do
        most = 5e9 / (2 * steps * layers * batch * hkv * dim * (4 if dtype == "f32" else 2))
        return dict(kind=kind, layers=layers, batch=batch, q_heads=hq, kv_heads=hkv, dim=dim,
                    dtype=dtype, budget=min(_log(rng, 64, 2048), int(most)),
                    ratio=rng.choice([1.0, 4.0, 8.0]), steps=steps)
    hq, hkv, dim, window, dtype = (32, 8, 128, 32, "bf16") if kind == "attn" else rng.choice(_SHAPES)
    layers = 1 if kind in ("layer", "select") else rng.choice([1, 4, 8, 16, 32])
    batch = rng.choice([1, 2, 4])
    seq = _log(rng, 512, 32768)
    # at most 4 GB of keys and values and, for the less common shapes, 1e10 multiply-adds of
    # scoring (about layers_d64_avg's)
    elem = 4 if dtype == "f32" else 2
    common = dtype == "bf16" and dim == 128 and hq // hkv * window in (128, 256)
    while layers > 1 and not common and 2048 * layers * batch * hq * window * dim > 1e10:
        layers //= 2
    most = 4e9 / (2 * layers * batch * hkv * dim * elem)
    if not common:
        most = min(most, 1e10 / (layers * batch * hq * window * dim))
    seq = max(256, min(seq, int(most)))
    pool, pk = rng.choice([("max", 7), ("max", 7), ("avg", 5), ("max", 13), ("none", 1)])
    return dict(kind=kind, layers=layers, batch=batch, q_heads=hq, kv_heads=hkv, dim=dim,
                seq=seq, window=window, pool=pool, pool_kernel=pk, dtype=dtype,
                budget=max(window, min(_log(rng, 64, 2048), seq // 2)),
                ratio=1.0 if layers == 1 else rng.choice([1.0, 4.0, 8.0]))


# ------------------------------------------------------------------ inputs


def _gen(seed, tag):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + tag) & ((1 << 62) - 1))
    return g


def _randn(shape, dtype, seed, tag):
    return torch.randn(shape, dtype=dtype, device=DEV, generator=_gen(seed, tag))


def _budgets(c):
    """A mid-depth bump of sensitivities (the shape of the paper's profiles) through the
    allocator; the same for every seed, as a program keeps one profile per model."""
    L = c["layers"]
    sens = [0.05 + math.exp(-((l - 0.4 * L) / (0.15 * L + 0.5)) ** 2) for l in range(L)]
    return R.ripple_alloc_budgets(sens, c["ratio"], math.inf, c["budget"] * L)


def _channel_scale(c, seed):
    x = torch.randn((c["layers"], 1, c["kv_heads"], 1, c["dim"]), device=DEV, generator=_gen(seed, 1))
    return torch.exp(0.5 * x).to(_DT[c["dtype"]])


def _prefill(c, seed):
    shape = (c["layers"], c["batch"], c["kv_heads"], c["seq"], c["dim"])
    dt = _DT[c["dtype"]]
    scale = _channel_scale(c, seed)
    k = _randn(shape, dt, seed, 2).mul_(scale)
    k[:, :, :, :4] += 3 * scale
    v = _randn(shape, dt, seed, 3)
    q = _randn((c["layers"], c["batch"], c["q_heads"], c["window"], c["dim"]), dt, seed, 4).mul_(2)
    return q, k, v


def _arena(rows, dtype, dim):
    """One buffer for all layers' caches (rows[l] cache rows in layer l) and its per-layer
    flat ranges, as a server that lays its caches out once keeps them."""
    flat = torch.zeros(sum(rows) * dim, dtype=dtype, device=DEV)
    return flat, flat.split([n * dim for n in rows])


def _prepare_compress(c, seed):
    q, k, v = _prefill(c, seed)
    L, B, H, D, dt = c["layers"], c["batch"], c["kv_heads"], c["dim"], _DT[c["dtype"]]
    budgets = _budgets(c)
    keep = [R.ripple_keep_count(b, c["seq"], c["window"]) for b in budgets]
    desc = R.layer_desc(B, c["q_heads"], H, D, c["seq"], c["window"], c["pool_kernel"], c["pool"], dt)
    rows = [B * H * n for n in keep]
    kf, ks = _arena(rows, dt, D)
    vf, vs = _arena(rows, dt, D)
    # index ranges start on 16-byte boundaries
    pad = [(n + 3) // 4 * 4 for n in rows]
    idx = torch.zeros(sum(pad), dtype=torch.int32, device=DEV)
    ix = [x[:n] for x, n in zip(idx.split(pad), rows)]
    ks = [x.view(B, H, n, D) for x, n in zip(ks, keep)]
    vs = [x.view(B, H, n, D) for x, n in zip(vs, keep)]
    s = dict(desc=desc, budgets=budgets, q=list(q), k=list(k), v=list(v), ks=ks, vs=vs, ix=ix,
             status=torch.zeros(1, dtype=torch.int32, device=DEV))
    s["out"] = {"k": kf.view(_INT[c["dtype"]]), "v": vf.view(_INT[c["dtype"]]), "idx": idx}
    if c["kind"] in ("layers", "attn"):
        s["tables"] = R.CompressTables(s["q"], s["k"], s["v"], ks, vs, ix)
    if c["kind"] == "layers":
        need = R.ripple_compress_layers_workspace_bytes(desc, L)
    elif c["kind"] == "attn":
        need = R.ripple_compress_layers_attn_workspace_bytes(desc, L)
        o = torch.zeros((L, B, c["q_heads"], c["window"], D), device=DEV)
        s["o_win"] = list(o)
        s["out"]["o_win"] = o
    else:
        need = R.ripple_compress_workspace_bytes(desc)
        votes = torch.zeros((B, H, c["seq"] - c["window"]), device=DEV)
        if c["kind"] == "layer":
            s["out"]["votes"] = votes
        else:
            # heavy-tailed votes, as the window softmax gives them
            torch.exp(1.5 * _randn(votes.shape, torch.float32, seed, 5), out=votes)
            votes.mul_(1e-3)
        s["votes"] = votes
    s["ws"] = torch.empty(need, dtype=torch.uint8, device=DEV)
    return s


def _decode_lens(c):
    return [max(32, b) for b in _budgets(c)]


def _prepare_decode(c, seed):
    L, B, Hq, H, D, dt = (c["layers"], c["batch"], c["q_heads"], c["kv_heads"], c["dim"],
                          _DT[c["dtype"]])
    lens, steps = _decode_lens(c), c["steps"]
    caps = [n + 64 for n in lens]
    scale = _channel_scale(c, seed)
    kf, vf = (_randn((sum(caps) * B * H * D,), dt, seed, tag) for tag in (10, 11))
    kc, vc = ([x.view(B, H, n, D) for x, n in zip(f.split([n * B * H * D for n in caps]), caps)]
              for f in (kf, vf))
    for l in range(L):
        kc[l].mul_(scale[l])
    caches = {"k": kf.view(_INT[c["dtype"]]), "v": vf.view(_INT[c["dtype"]])}
    kn = _randn((steps, L, B, H, D), dt, seed, 6).mul_(scale.view(1, L, 1, H, D))
    vn = _randn((steps, L, B, H, D), dt, seed, 7)
    q = _randn((steps, L, B, Hq, D), dt, seed, 8).mul_(2)
    # the prompt's lengths, to which the loop goes back (another sample of the same prompt)
    start = torch.tensor(lens, dtype=torch.int32, device=DEV)
    s = dict(start=start, lens=start.clone(), steps=steps, q=q, kn=kn, vn=vn, kc=kc, vc=vc,
             status=torch.zeros(1, dtype=torch.int32, device=DEV))
    if c["kind"] == "loop":
        loop = LayerDecodeLoop(
            kc, vc, s["lens"], Hq, lambda l: (q[0, l:l + 1], kn[0, l:l + 1], vn[0, l:l + 1]),
            lambda l, out: None)
        loop.issue_step()
        loop.capture()
        s["loop"] = loop
        s["ret"] = {"out": loop.out, "lens": s["lens"], **caches}
    else:
        s["desc"] = R.decode_desc(L, B, Hq, H, D, dt)
        s["tables"] = R.DecodeTables(kc, vc)
        s["ws"] = torch.empty(R.ripple_decode_workspace_bytes(s["desc"], caps),
                              dtype=torch.uint8, device=DEV)
        s["o"] = torch.zeros((steps, L, B, Hq, D), device=DEV)
        s["ret"] = {"out": s["o"], "lens": s["lens"], **caches}
    return s


def _prepare_perturb(c, seed):
    shape = (c["batch"], c["kv_heads"], c["seq"], c["dim"])
    v = _randn(shape, _DT[c["dtype"]], seed, 2)
    eps = _randn(shape[:2] + (c["seq"] - c["window"], c["dim"]), torch.float32, seed, 3)
    return dict(v=v, eps=eps, end=c["seq"] - c["window"], out=torch.zeros_like(v))


def _kl_logits(c, seed):
    p = _randn((c["pos"], c["vocab"]), torch.float32, seed, 2).mul_(2.5)
    at = torch.randint(0, c["vocab"], (c["pos"], 4), device=DEV, generator=_gen(seed, 3))
    p.scatter_add_(1, at, torch.full(at.shape, 12.0, device=DEV))
    q = _randn((c["sets"], c["pos"], c["vocab"]), torch.float32, seed, 4)
    sigma = torch.linspace(0.02, 0.3, c["sets"], device=DEV)
    q.mul_(sigma.view(-1, 1, 1)).add_(p)
    return p.to(_DT[c["dtype"]]), q.to(_DT[c["dtype"]])


def _prepare_kl(c, seed):
    p, q = _kl_logits(c, seed)
    ws = torch.empty(R.ripple_window_kl_workspace_bytes(c["sets"], c["pos"], c["vocab"]),
                     dtype=torch.uint8, device=DEV)
    return dict(p=p, q=q, ws=ws, d=torch.zeros(c["sets"], device=DEV),
                kl=torch.zeros((c["sets"], c["pos"]), device=DEV),
                status=torch.zeros(1, dtype=torch.int32, device=DEV))


def prepare(case, seed):
    c = case
    make = {"loop": _prepare_decode, "decode": _prepare_decode, "perturb": _prepare_perturb,
            "kl": _prepare_kl}.get(c["kind"], _prepare_compress)
    s = make(c, seed)
    s["kind"] = c["kind"]
    return s


# ------------------------------------------------------------------ the calls


def run(s):
    kind = s["kind"]
    if kind == "layers":
        R.ripple_compress_layers(s["desc"], s["budgets"], s["tables"], s["ws"], dev_status=s["status"])
        return s["out"]
    if kind == "attn":
        R.ripple_compress_layers_attn(s["desc"], s["budgets"], s["tables"], s["o_win"], s["ws"],
                                      dev_status=s["status"])
        return s["out"]
    if kind == "layer":
        R.ripple_compress_layer(s["desc"], s["budgets"][0], s["q"][0], s["k"][0], s["v"][0],
                                s["ks"][0], s["vs"][0], s["ix"][0], s["ws"],
                                scores_out=s["votes"], dev_status=s["status"])
        return s["out"]
    if kind == "select":
        R.ripple_select_layer(s["desc"], s["budgets"][0], s["votes"], s["k"][0], s["v"][0],
                              s["ks"][0], s["vs"][0], s["ix"][0], s["ws"], dev_status=s["status"])
        return s["out"]
    if kind == "loop":
        s["lens"].copy_(s["start"])
        s["loop"].replay()
        return s["ret"]
    if kind == "decode":
        s["lens"].copy_(s["start"])
        for t in range(s["steps"]):
            R.ripple_decode_attn(s["desc"], s["q"][t], s["kn"][t], s["vn"][t], s["tables"],
                                 s["lens"], s["o"][t], s["ws"], dev_status=s["status"])
        return s["ret"]
    if kind == "perturb":
        R.ripple_perturb_values(s["v"], s["eps"], 0.05, 0, s["end"], v_out=s["out"])
        return s["out"]
    R.ripple_window_kl(s["p"], s["q"], s["ws"], s["d"], kl_out=s["kl"], dev_status=s["status"])
    return {"d": s["d"], "kl": s["kl"]}


# ------------------------------------------------------------------ what a pass cannot do without


def work(case):
    c = case
    e = 4 if c["dtype"] == "f32" else 2
    if c["kind"] == "kl":
        return {"bytes": (c["sets"] + 1) * c["pos"] * c["vocab"] * e, "flops": 0}
    if c["kind"] == "perturb":
        rows = c["batch"] * c["kv_heads"] * c["seq"]
        part = c["batch"] * c["kv_heads"] * (c["seq"] - c["window"])
        return {"bytes": rows * c["dim"] * 2 * e + part * c["dim"] * 4, "flops": 0}
    L, B, Hq, H, D = c["layers"], c["batch"], c["q_heads"], c["kv_heads"], c["dim"]
    if c["kind"] in ("loop", "decode"):
        lens, b, f = _decode_lens(c), 0, 0
        for t in range(c["steps"]):
            rows = sum(n + t + 1 for n in lens) * B * H
            b += 2 * rows * D * e + L * B * (Hq * D * (e + 4) + 4 * H * D * e)
            f += 4 * rows * D * (Hq // H)
        return {"bytes": b, "flops": f}
    T, W, units = c["seq"], c["window"], B * H
    keep = sum(R.ripple_keep_count(x, T, W) for x in _budgets(c))
    out = units * keep * (2 * D * e + 4)  # kept rows and their positions written
    if c["kind"] == "select":  # votes, and the kept rows read
        return {"bytes": out + units * (4 * (T - W) + 2 * keep * D * e), "flops": 0}
    b = out + L * units * T * D * e + L * B * Hq * W * D * e
    f = 2 * L * B * Hq * W * T * D
    if c["kind"] == "attn":  # every value once, and the window rows' output
        return {"bytes": b + L * units * T * D * e + 4 * L * B * Hq * W * D, "flops": 2 * f}
    if c["kind"] == "layer":
        b += 4 * units * (T - W)
    return {"bytes": b + units * keep * D * e, "flops": f}


def tolerance(case):
    k = case["kind"]
    if k == "select":
        return "exact"  # votes are given: the same tokens, bytes for bytes
    if k in ("layers", "layer", "attn"):
        # votes: fp32 sums of probabilities (2.5e-7 from 64 bits here, up to a few times that
        # for longer rows); o_win: probabilities rounded to bf16 (1.5e-3); kept places:
        # near-ties at the threshold
        return {"rel": 6e-3 if k == "attn" else 3e-6, "differ": 0.01}
    if k in ("loop", "decode"):
        return {"rel": 2e-6}  # 4e-7 from 64 bits
    if k == "perturb":
        # fp32 arithmetic, rounded once to the cache's type: at a rounding midpoint one step
        # of bf16 (2^-8 of the value)
        return {"rel": 6e-5, "max": 8e-3} if case["dtype"] == "bf16" else {"rel": 1e-6}
    return {"rel": 3e-5}  # 7e-6 from 64 bits: a divergence is a small difference of large sums


# ------------------------------------------------------------------ the same in 64 bits


def _votes64(c, q, k, v=None):
    """Votes of one unit's prefix keys, and the window rows' outputs with v; q [G*w][d]."""
    T, W = c["seq"], c["window"]
    x = (q.double() @ k.double().T) / math.sqrt(c["dim"])
    last = T - W + torch.arange(q.shape[0], device=q.device) % W
    x.masked_fill_(torch.arange(T, device=q.device)[None, :] > last[:, None], -math.inf)
    p = torch.softmax(x, 1)
    return p.sum(0)[:T - W], None if v is None else p @ v.double()


def exact(case, seed):
    c = case
    if c["kind"] == "kl":
        p, q = _kl_logits(c, seed)
        lp = torch.log_softmax(p.double(), 1)
        kl = torch.stack([(lp.exp() * (lp - torch.log_softmax(x.double(), 1))).sum(1) for x in q])
        return {"d": kl.mean(1), "kl": kl}
    if c["kind"] == "perturb":
        s = _prepare_perturb(c, seed)
        out = s["v"].double()
        head = out[:, :, :s["end"]]
        head += 0.05 * head.norm(dim=3, keepdim=True) * s["eps"].double()
        return out
    if c["kind"] in ("loop", "decode"):
        s = _prepare_decode(dict(c, kind="decode"), seed)
        lens, H = _decode_lens(c), c["kv_heads"]
        o = torch.zeros(s["o"].shape, dtype=torch.float64, device=DEV)
        for l, n in enumerate(lens):
            k, v = s["kc"][l].double(), s["vc"][l].double()
            for t in range(c["steps"]):
                k[:, :, n + t], v[:, :, n + t] = s["kn"][t, l].double(), s["vn"][t, l].double()
                q = s["q"][t, l].double().view(c["batch"], H, -1, c["dim"])
                x = q @ k[:, :, :n + t + 1].transpose(2, 3) / math.sqrt(c["dim"])
                o[t, l] = (torch.softmax(x, 3) @ v[:, :, :n + t + 1]).reshape(o[t, l].shape)
        if c["kind"] == "loop":
            return {"out": [x[None] for x in o[0]], "lens": None, "k": None, "v": None}
        return {"out": o, "lens": None, "k": None, "v": None}
    if c["kind"] not in ("layer", "attn"):
        return None  # positions and byte copies
    q, k, v = _prefill(c, seed)
    L, B, H = c["layers"], c["batch"], c["kv_heads"]
    qu = q.view(L, B, H, -1, c["dim"])
    got = [_votes64(c, qu[l, b, h], k[l, b, h], v[l, b, h] if c["kind"] == "attn" else None)
           for l in range(L) for b in range(B) for h in range(H)]
    out = {"k": None, "v": None, "idx": None}
    if c["kind"] == "layer":
        out["votes"] = torch.stack([x[0] for x in got]).view(B, H, -1)
    else:
        out["o_win"] = torch.stack([x[1] for x in got]).view(L, B, c["q_heads"], c["window"], -1)
    return out
