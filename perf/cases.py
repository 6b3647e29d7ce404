"""The work that is timed: what a program that serves a model with a compressed KV cache asks of this library.

A case is one dict of plain values.  Its ``kind`` says which calls one pass makes:

  decode   one decode step: sc_decode_attn for each of L layers.  ``graph``: the layers are a dependent chain
           (layer l+1's query is layer l's output) replayed from a CUDA graph, as a low-batch decode loop runs it;
           else eager calls, one independent query per layer.  ``count`` false: exact attention over a raw cache.
  turn     the whole path for one layer with the convenience wrappers: chunk -> compress -> one decode step
  prompt   the end of a prefill: sc_chunk, then every layer's cache is compressed.  ``one_launch``: all layers
           exist and go through sc_compress_layers; else one sc_compress per layer, as a layer-by-layer prefill does
  prefill  sc_prefill_attn: a block of m queries per head over each of L layers' cores
  spec     one round of speculative decoding over L layers: m draft tokens verified by sc_prefill_attn, then the
           lengths are rolled back and the m tokens are accepted with sc_append_layers, one call per token

Sizes are those of the repository's own workloads (``synth.config``) and tests, odd ones beside them; ``draw`` covers the ranges between.
"""
from __future__ import annotations

import math

import torch

from paper_2603_14303_b200 import binding as sc
from paper_2603_14303_b200 import synth

DEV = "cuda"
_DEFAULT = dict(B=1, n=32768, Hkv=8, G=4, d=128, dtype="bf16", L=1, kept=0.26, cap_div=2, spread=0.0, count=True,
                graph=False, gap="poisson", gap_mean=20.0, c_max=8, ratio=0.0, token_major=False, one_launch=False,
                m=1, causal=False)
# the parameters each kind reads (a case holds these and no others)
_USED = {
    "decode": "B n Hkv G d dtype L kept cap_div spread count graph",
    "turn": "B n Hkv G d dtype gap gap_mean c_max ratio",
    "prompt": "B n Hkv d dtype L cap_div gap gap_mean c_max ratio token_major one_launch",
    "prefill": "B n Hkv G d dtype L kept cap_div spread m causal",
    "spec": "B n Hkv G d dtype L kept cap_div spread m",
}
_MAX_BYTES = 5.0e9     # of a drawn case: below the largest listed one (32 layers of a 32K-token prompt, 5.4 GB)
_MAX_FLOPS = 2.5e11    # of a drawn case: below the largest listed one (512 queries per head over 4 layers)


def _case(kind, **kw):
    c = {"kind": kind, **{k: _DEFAULT[k] for k in _USED[kind].split()}}
    assert set(kw) <= set(c) | {"name"}, set(kw) - set(c)
    c.update(kw)
    return c


def listed():
    return [
        # one attention call over the cores of a 2K-token context: a short chat, pure latency
        _case("decode", name="decode_2k", n=2048, kept=0.25),
        # a whole decode step of a 32-layer model at 32K context, batch 1
        _case("decode", name="decode_32k_chain", L=32, graph=True),
        # the same with 7 query heads per KV head, 4 KV heads, 128K context, 28 layers
        _case("decode", name="decode_128k_g7_chain", n=131072, Hkv=4, G=7, L=28, graph=True),
        # batched serving: 16 sequences of up to 16K tokens at different points of their generation
        _case("decode", name="decode_16x16k", B=16, n=16384, L=4, kept=0.28, spread=0.5),
        # layers whose cache is left uncompressed: exact attention over 64K raw rows, batch 4, odd length
        _case("decode", name="decode_raw_4x64k", B=4, n=65531, L=2, kept=1.0, cap_div=1, count=False),
        # a short prompt end to end, one layer: chunk, compress, first decode step (latency, many small launches)
        _case("turn", name="turn_2k", n=2048, gap_mean=24.0, c_max=6),
        # the same path in float32, at an odd length
        _case("turn", name="turn_f32_8k", n=8191, dtype="f32"),
        # end of a 32K prefill: 32 layers compressed at once
        _case("prompt", name="prompt_32k", L=32, one_launch=True),
        # batched prefill of ragged text (lognormal chunk lengths), token-major storage, layer by layer
        _case("prompt", name="prompt_16x16k", B=16, n=16384, L=2, gap="lognormal", gap_mean=18.0, token_major=True),
        # text with long chunks (mean 128 tokens, up to 256), batch 4 at 64K, compressed eightfold
        _case("prompt", name="prompt_4x64k_long", B=4, n=65536, L=1, gap_mean=128.0, ratio=8.0),
        # a chunk of 512 prompt tokens attends to a compressed 32K past and to itself
        _case("prefill", name="prefill_512", m=512, L=4, causal=True),
        # 8 draft tokens verified and accepted, 8 layers
        _case("spec", name="spec_8", m=8, L=8),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case: sizes log-uniform over the listed ranges, odd ones included, within the largest listed cost."""
    kind = rng.choice(["decode", "decode", "turn", "prompt", "prompt", "prefill", "spec"])
    Hkv, G = rng.choice([(8, 4), (8, 4), (4, 7)])
    text = dict(gap="poisson", gap_mean=round(_log(rng, 8, 128), 1), c_max=rng.choice([4, 6, 8]),
                ratio=rng.choice([0.0, 0.0, 4.0, 8.0]))
    if rng.random() < 0.3:
        text.update(gap="lognormal", gap_mean=18.0)
    cores = dict(kept=round(rng.uniform(0.12, 0.5), 3), cap_div=rng.choice([1, 2]))
    while True:
        B = rng.choice([1, 1, 2, 3, 4, 7, 16])
        n = int(_log(rng, 2048, 131072))
        if kind == "decode":
            graph = B <= 2 and rng.random() < 0.7
            c = _case(kind, B=B, n=n, Hkv=Hkv, G=G, graph=graph, L=rng.randint(8, 32) if graph else rng.randint(1, 4),
                      spread=0.5 if B > 1 else 0.0, **cores)
            if not graph and rng.random() < 0.2:
                c.update(kept=1.0, cap_div=1, count=False)
        elif kind == "turn":
            f32 = rng.random() < 0.4
            c = _case(kind, B=min(B, 2), n=int(_log(rng, 2048, 8192 if f32 else 32768)), Hkv=Hkv, G=G,
                      dtype="f32" if f32 else "bf16", **text)
        elif kind == "prompt":
            one = rng.random() < 0.5
            c = _case(kind, B=B, n=n, Hkv=Hkv, L=rng.randint(4, 32) if one else rng.randint(1, 3), one_launch=one,
                      token_major=rng.random() < 0.5, cap_div=1, **text)
        elif kind == "prefill":
            c = _case(kind, B=min(B, 4), n=max(n, 8192), Hkv=Hkv, G=G, m=int(_log(rng, 16, 1024)), L=rng.randint(1, 8),
                      causal=rng.random() < 0.5, **cores)
        else:
            c = _case(kind, B=min(B, 4), n=n, Hkv=Hkv, G=G, m=rng.randint(2, 16), L=rng.randint(2, 16), **cores)
        w = work(c)
        if w["bytes"] <= _MAX_BYTES and w["flops"] <= _MAX_FLOPS and c["B"] * c["n"] <= 262144:
            return c


# ------------------------------------------------------------------------------------------ what a pass needs


def _esize(c):
    return 2 if c["dtype"] == "bf16" else 4


def _rows(c):
    """Expected cores of a head."""
    return c["kept"] * c["n"] * (1.0 - c["spread"] / 2) + (c["m"] / 2 if c.get("causal") else 0)


def _text_kept(c):
    """Expected kept fraction of the generated text: distinct centroids of a chunk, plus its delimiter."""
    ln = max(c["gap_mean"], 1.0) * (1.35 if c["gap"] == "lognormal" else 1.0)
    if c["ratio"]:
        seeds = [max(1.0, (ln + 1.0) / c["ratio"] - 1.0)]
    else:
        seeds = range(1, c["c_max"] + 1)
    distinct = sum(s * (1.0 - (1.0 - 1.0 / s) ** ln) for s in seeds) / len(seeds)
    return (distinct + 1.0) / (ln + 1.0)


def _compress_work(c, L):
    tokens, d = c["B"] * c["Hkv"] * c["n"] * L, c["d"]
    f = min(_text_kept(c), 1.0)
    row = 2 * d * _esize(c)
    return tokens * (row + f * (row + 4)) + 8 * c["B"] * c["n"], tokens * d * (c["gap_mean"] + 2)


def work(case):
    c, kind, d = case, case["kind"], case["d"]
    if kind == "prompt":
        b, f = _compress_work(c, c["L"])
        return {"bytes": b, "flops": f}
    heads = c["B"] * c["Hkv"]
    if kind == "turn":
        b, f = _compress_work(c, 1)
        rows = min(_text_kept(c), 1.0) * c["n"]
        b += heads * (rows * (2 * d * _esize(c) + 4) + 2 * c["G"] * d * _esize(c))
        return {"bytes": b, "flops": f + 4 * heads * c["G"] * rows * d}
    m = c.get("m", 1)
    row = 2 * d * _esize(c) + (4 if c.get("count", True) else 0)
    b = c["L"] * heads * (_rows(c) * row + 2 * c["G"] * m * d * _esize(c))
    if kind == "spec":
        b += c["L"] * heads * m * 2 * (row + 2 * d * _esize(c))
    return {"bytes": b, "flops": 4 * c["L"] * heads * c["G"] * m * _rows(c) * d}


def tolerance(case):
    # Against 64-bit evaluations of the same inputs every kind shows 1.4e-3 to 1.7e-3 in bf16 (the rounding of the
    # result) and 2.6e-7 in float32 (sums of up to 2K terms): four times that, for two implementations.  Counts,
    # lengths and assignments are whole numbers and agree exactly.
    return {"rel": 6.5e-3} if case["dtype"] == "bf16" else {"rel": 1.5e-6}


# ------------------------------------------------------------------------------------------ inputs


def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1000003 + salt * 7919 + 11) & 0x7FFFFFFFFFFFFFFF)
    return g


def _extra(c):
    """Rows behind the compressed past: the block's own tokens, or room for accepted drafts."""
    return 32 if c["kind"] == "spec" else c["m"] if c.get("causal") else 0


def _cap(c):
    return max(c["n"] // c["cap_div"], 1) + _extra(c)


def _cores(c, seed, layer):
    """Semantic cores as sc_compress leaves them: unit-scale keys, means of N(0, 1) values, counts >= 1 whose mean is
    1 / kept, heads of slightly different lengths (sequences of a batch up to ``spread`` shorter), behind them the
    block's own tokens with count 1 where it attends to itself; rows past a head's end are zero."""
    g = _gen(seed, 1 + layer)
    B, H, d, cap = c["B"], c["Hkv"], c["d"], _cap(c)
    part = 1.0 - c["spread"] * torch.rand((B, 1), generator=_gen(seed, 0), device=DEV)
    if c.get("count", True):
        part = part * (1.0 + 0.02 * torch.randn((B, H), generator=g, device=DEV))
    ln = (part.expand(B, H) * (c["kept"] * c["n"])).round().int().clamp(1, cap - _extra(c)).contiguous()
    past = ln
    if c.get("causal"):
        ln = ln + c["m"]
    live = torch.arange(cap, device=DEV).view(1, 1, cap) < ln.unsqueeze(2)
    mean = max(1.0 / c["kept"] - 1.0, 0.0) if c["kept"] < 1 else 0.0
    u = torch.rand((B, H, cap), generator=g, device=DEV).clamp_(min=1e-7)
    count = torch.where(live, 1 + torch.floor(-mean * torch.log(u) + 0.5), 0.0).int()
    count[live & (torch.arange(cap, device=DEV).view(1, 1, cap) >= past.unsqueeze(2))] = 1
    k = torch.empty((B, H, cap, d), dtype=_dtype(c), device=DEV)
    v = torch.empty_like(k)
    for b in range(B):      # one sequence at a time: the float32 intermediates stay small
        kb = torch.randn((H, cap, d), generator=g, device=DEV)
        k[b] = torch.where(live[b].unsqueeze(2), kb / kb.norm(dim=2, keepdim=True), 0.0)
        vb = torch.randn((H, cap, d), generator=g, device=DEV) / count[b].clamp(min=1).sqrt().unsqueeze(2)
        v[b] = torch.where(live[b].unsqueeze(2), vb, 0.0)
    return sc.CompressedLayer(k, v, count, ln)


def _text(c, seed):
    gap = ("poisson", c["gap_mean"]) if c["gap"] == "poisson" else ("lognormal", c["gap_mean"], 0.8, 256)
    cen = ("ratio", c["ratio"]) if c["ratio"] else ("uniform", c["c_max"])
    w = synth.Workload("case", B=c["B"], n=c["n"], L=c.get("L", 1), Hkv=c["Hkv"], Hq=c["Hkv"] * c.get("G", 4), d=c["d"],
                       gap=gap, centroids=cen, seed=seed & 0x7FFFFFFF, dtype=c["dtype"])
    ids, run_id, run_lens = synth.token_ids(w)
    return w, ids.to(DEV), run_id, run_lens


def _kv(c, w, layer, run_id, run_lens):
    K, V = synth.layer_kv(w, layer, run_id, run_lens, device=DEV)
    if c.get("token_major"):   # [B, n, Hkv, d] storage seen head-major, as an attention layer writes it
        K, V = (t.transpose(1, 2).contiguous().transpose(1, 2) for t in (K, V))
    return K, V


def _stacked(s, core_k, core_v, count, core_len):
    """One buffer per field for all layers (returned whole); the layers are its slices."""
    s["cores"] = {"core_k": core_k, "core_v": core_v, "count": count, "core_len": core_len}
    s["layers"] = [sc.CompressedLayer(*row) for row in zip(core_k, core_v, count, core_len)]


def _randn(shape, g, dt):
    return torch.randn(shape, generator=g, device=DEV).to(dt)


def prepare(case, seed):
    c, kind, dt = case, case["kind"], _dtype(case)
    B, H, d, n = c["B"], c["Hkv"], c["d"], c["n"]
    s = {"case": c}
    if kind in ("turn", "prompt"):
        w, s["ids"], run_id, run_lens = _text(c, seed)
        layers = [_kv(c, w, l, run_id, run_lens) for l in range(c.get("L", 1))]
        s["K"], s["V"] = [k for k, _ in layers], [v for _, v in layers]
        cap = n if kind == "turn" else max(n // c["cap_div"], 1)
        rows = (len(layers), B, H, cap)
        _stacked(s, torch.zeros((*rows, d), dtype=dt, device=DEV), torch.zeros((*rows, d), dtype=dt, device=DEV),
                 torch.zeros(rows, dtype=torch.int32, device=DEV), torch.zeros(rows[:3], dtype=torch.int32, device=DEV))
        s["tau"] = w.tau
        if kind == "turn":
            s["q"] = synth.queries(w, 0, 0, device=DEV)
            s["ws"] = sc.compress_workspace(B, H, n, DEV)
            s["dws"] = sc.decode_workspace(B, w.Hq, H, d, cap, DEV)
        elif c["one_launch"]:
            s["ws"] = sc.compress_layers_workspace(c["L"], B, H, n, DEV)
        else:
            s["ws"] = sc.compress_workspace(B, H, n, DEV)
        return s
    Hq = H * c["G"]
    s["layers"] = [_cores(c, seed, l) for l in range(c["L"])]
    cap = _cap(c)
    g = _gen(seed, 1009)
    if kind == "decode":
        s["ws"] = sc.decode_workspace(B, Hq, H, d, cap, DEV)
        s["q"] = [_randn((B, Hq, d), g, dt) for _ in range(1 if c["graph"] else c["L"])]
        s["out"] = [torch.zeros((B, Hq, d), dtype=dt, device=DEV) for _ in range(c["L"])]
        if c["graph"]:
            _chain(s)          # once outside capture, as any capture is warmed up
            torch.cuda.synchronize()
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"]):
                _chain(s)
        return s
    m = c["m"]
    s["q"] = [_randn((B, Hq, m, d), g, dt) for _ in range(c["L"])]
    s["out"] = torch.zeros((c["L"], B, Hq, m, d), dtype=dt, device=DEV)
    if kind == "spec":
        y = s["layers"]
        _stacked(s, *(torch.stack([getattr(r, k) for r in y]) for k in ("core_k", "core_v", "count", "core_len")))
        # draft tokens: mostly ordinary ids, a delimiter every few tokens; keys around a few directions per head
        ids = torch.randint(1000, 20000, (m, B), generator=g, device=DEV, dtype=torch.int32)
        ids[m // 2] = synth.DELIMS[0]
        s["ids"] = ids
        near = torch.randint(0, 3, (c["L"], m, B, H), generator=g, device=DEV)
        cen = torch.randn((3, d), generator=g, device=DEV)
        cen = cen / cen.norm(dim=1, keepdim=True)
        s["k_new"] = (cen[near] + 0.15 / math.sqrt(d) * torch.randn((c["L"], m, B, H, d), generator=g, device=DEV)).to(dt)
        s["v_new"] = _randn((c["L"], m, B, H, d), g, dt)
        s["len0"] = s["cores"].pop("core_len")
        s["len"] = s["len0"].clone()
        s["tail"] = torch.zeros_like(s["len0"])
        s["attn"] = torch.zeros_like(s["len0"])
        s["tables"] = [sc.append_table([(s["k_new"][l, t], s["v_new"][l, t], y.core_k, y.core_v, y.count, s["len"][l],
                                         s["tail"][l], s["attn"][l]) for l, y in enumerate(s["layers"])]) for t in range(m)]
    return s


# ------------------------------------------------------------------------------------------ one pass


def _chain(s):
    x = s["q"][0]
    for y, o in zip(s["layers"], s["out"]):
        x = sc.decode_attn(x, y, out=o, workspace=s["ws"], flags=sc.SC_FLAG_OVERLAP_CHAIN)


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "decode":
        if c["graph"]:
            s["graph"].replay()
        else:
            for q, y, o in zip(s["q"], s["layers"], s["out"]):
                sc.decode_attn(q, y, out=o, workspace=s["ws"], use_count=c["count"])
        return s["out"]
    if kind == "turn":
        plan = sc.chunk(s["ids"], synth.DELIMS)
        y = sc.compress(s["K"][0], s["V"][0], plan, s["tau"], workspace=s["ws"], out=s["layers"][0])
        o = sc.decode_attn(s["q"], y, workspace=s["dws"])
        return {"attn": o, **s["cores"]}
    if kind == "prompt":
        plan = sc.chunk(s["ids"], synth.DELIMS)
        if c["one_launch"]:
            sc.sc_compress_layers(s["K"], s["V"], plan, s["tau"], s["layers"], s["ws"], plan.status)
        else:
            for K, V, y in zip(s["K"], s["V"], s["layers"]):
                sc.compress(K, V, plan, s["tau"], workspace=s["ws"], out=y)
        return s["cores"]
    if kind == "prefill":
        for q, y, o in zip(s["q"], s["layers"], s["out"]):
            sc.prefill_attn(q, y, out=o, causal=c["causal"])
        return s["out"]
    for q, y, o in zip(s["q"], s["layers"], s["out"]):
        sc.prefill_attn(q, y, out=o)
    s["len"].copy_(s["len0"])
    s["tail"].zero_()
    k0 = s["k_new"][0, 0]
    for ids, table in zip(s["ids"], s["tables"]):
        sc.sc_append_layers(table, k0, ids, synth.DELIMS, sc.SC_MAX_CHUNK_LEN, 0.7, s["layers"][0].core_k.shape[2])
    return {"attn": s["out"], "core_len": s["len"], "tail_len": s["tail"], "attn_len": s["attn"], **s["cores"]}
