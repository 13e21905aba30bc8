"""The work that programs built on this library have it do, as measurable cases.

A scene query runs: query preparation, relevance scores, pruning, budgets and token selection,
(optionally the merge of the unselected tokens and the predictor's features), ragged packing, the
decoder prefill over the packed batch, and the decode step over its KV cache.  The cases take each
of these through the public entry points, from the smallest call to the 400-tile query:

  kind "scene"      ScenePipeline.run(prefill=False): select (and merge) and pack one scene
  kind "features"   abi.tile_features on a selected scene's kept tiles
  kind "prefill"    abi.prefill_layers on packed sequences, with the KV cache and the logits
  kind "prefix"     abi.prefill_shared_prefix: the system prompt once, the suffixes over its cache
  kind "attention"  abi.attention_varlen on packed q, k, v
  kind "decode"     ScenePipeline-style decode step: abi.decode_step with logits
  kind "query"      a whole scene query: select, pack, prefill, last-token logits

Shapes are the repository's own: 576-token tiles (24 x 24) of 4096-wide tokens, S = 35 system and
Q = 24 query tokens, M = 8 background terms, budgets {72, 144, 288, 432, 576}, the 7B decoder shape
(d 4096, 32 heads x 128, FFN 11008, vocabulary 32000) and the small test decoder (d 256, head 64).
Blocks of a few decoder layers stand for the 32-layer stack, whose layers are alike.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_2609_29029_gb300 import DeviceModel, ScenePipeline, abi

DEV = "cuda"
S_SYS, Q_IDS, VOCAB = 35, 24, 32000
BUDGETS = (72, 144, 288, 432, 576)
ALPHA_POS = (0.86, 0.87, 0.875, 0.877, 0.878)
ALPHA_NEG = (0.50, 0.68, 0.84, 0.868, 0.89)
ENERGY = (0.28, 0.40, 0.62, 0.82, 1.00)
PLANTED, DISTRACTORS = 0.05, 0.18  # share of the tiles that hold the object / look a little like it
KEPT, MEAN_BUDGET = 0.18, 0.46     # what the 400-tile scene keeps, and of how many tokens (for work())


# ---------------------------------------------------------------------------------------- the cases

def listed():
    big = dict(d=4096, heads=32, ffn=11008, vocab=VOCAB)
    return [
        # the smallest call: four small fp32 tiles, where only latency and launches count
        dict(name="scene_tiny_f32", kind="scene", N=4, n_v=576, d=256, f32=True, M=8, S=35, Q=24, knn=6, merge=False),
        # one query over a 64-tile scene (the method's walkthrough size)
        dict(name="scene_64", kind="scene", N=64, n_v=576, d=4096, f32=False, M=8, S=35, Q=24, knn=6, merge=False),
        # one query over a 400-tile scene, up to the packed batch
        dict(name="scene_400", kind="scene", N=400, n_v=576, d=4096, f32=False, M=8, S=35, Q=24, knn=6, merge=False),
        # the same scene with the unselected tokens merged into contextual ones
        dict(name="scene_400_merge", kind="scene", N=400, n_v=576, d=4096, f32=False, M=8, S=35, Q=24, knn=6,
             merge=True),
        # the budget predictor's features of the kept tiles
        dict(name="features_400", kind="features", N=400, n_v=576, d=4096, f32=False, M=8, knn=6),
        # one kept tile at the smallest budget (72 + 59 rows), the interactive single-tile question
        dict(name="prefill_one_tile", kind="prefill", layers=2, seqs=1, extra=0, mix=0, **big),
        # the kept tiles of a 64-tile scene (17 sequences, about 4.3K rows)
        dict(name="prefill_scene_64", kind="prefill", layers=2, seqs=17, extra=0, mix=1, **big),
        # the same kind of batch (9 sequences) over a system prompt that is prefilled once
        dict(name="prefix_9_tiles", kind="prefix", layers=2, seqs=9, extra=0, mix=1, S=35, **big),
        # the first answer token of one tile
        dict(name="decode_1", kind="decode", layers=4, seqs=1, extra=0, mix=2, **big),
        # the first answer token of each of a 400-tile scene's kept tiles
        dict(name="decode_73", kind="decode", layers=4, seqs=73, extra=0, mix=1, **big),
        # attention alone on long sequences (several tiles asked about together)
        dict(name="attention_long", kind="attention", seqs=5, L=4096, ragged=False, heads=32, hd=128),
        # the whole query: 400 tiles, 32 layers, last-token logits
        dict(name="query_400", kind="query", N=400, layers=32, n_v=576, f32=False, M=8, S=35, Q=24, knn=6,
             merge=False, **big),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges: scene sizes, token grids, widths, types and options;
    batch sizes, lengths and decoder shapes."""
    kind = rng.choice(["scene", "scene", "features", "prefill", "prefill", "prefix", "decode", "decode", "attention"])
    if kind in ("scene", "features"):
        f32 = rng.random() < 0.25
        d = rng.choice([256, 1024, 2048, 4096])
        g = rng.choice([10, 14, 16, 24, 24, 24])
        n_v = g * g if kind == "features" or rng.random() < 0.6 else rng.randint(72, 600)
        c = dict(kind=kind, N=_log_int(rng, 4, 700 if not f32 else 300), n_v=n_v, d=d, f32=f32,
                 M=rng.choice([0, 3, 8, 8]), knn=rng.choice([0, 4, 6, 6]))
        if kind == "scene":
            c.update(S=rng.choice([0, 5, 35, 35]), Q=rng.randint(1, 40), merge=rng.random() < 0.4)
        return c
    if kind == "attention":
        L = _log_int(rng, 40, 4096)
        return dict(kind=kind, seqs=max(1, min(200, int(20000 * rng.uniform(0.1, 1.0) / L))), L=L,
                    ragged=rng.random() < 0.7, heads=rng.choice([4, 16, 32]), hd=rng.choice([64, 128, 128]))
    shape = rng.choice([dict(d=4096, heads=32, ffn=11008, vocab=VOCAB)] * 4 +
                       [dict(d=1024, heads=8, ffn=2816, vocab=4096), dict(d=256, heads=4, ffn=688, vocab=1000)])
    c = dict(kind=kind, layers=rng.randint(1, 3), extra=rng.choice([0, 0, rng.randint(1, 40)]),
             mix=rng.choice([0, 1, 1, 2]), **shape)
    if kind == "decode":
        c["seqs"] = _log_int(rng, 1, 150)
    else:
        c["seqs"] = _log_int(rng, 1, 40)
        if kind == "prefix":
            c["S"] = rng.choice([8, 35, 35, 60, 200])
    return c


# ---------------------------------------------------------------------------------------- inputs

def _gen(seed, *more):
    g = torch.Generator(device=DEV)
    s = seed * 1_000_003 + 17
    for m in more:
        s = s * 8191 + int(m)
    g.manual_seed(s % (1 << 62))
    return g


def _randn(gen, *shape, dtype=torch.float32, scale=1.0):
    x = torch.randn(*shape, dtype=dtype, device=DEV, generator=gen)
    return x if scale == 1.0 else x.mul_(scale)


def _policy(case):
    n_v = case["n_v"]
    C = sorted({max(1, c * n_v // 576) for c in BUDGETS})
    k = len(C)
    return SimpleNamespace(tau=0.37, C=tuple(C), alpha_pos=ALPHA_POS[:k], alpha_neg=ALPHA_NEG[:k], energy=ENERGY[:k],
                           lam=0.15, ctx_num=10 if case.get("merge") else 0, ctx_den=64)


def _scene(case, seed):
    """Vision tokens N(0, 1); the tiles that hold the object add the query's direction on a patch of
    tokens, look-alikes add less of it and a background direction.  The embedding rows of the query
    and of the background terms point along those directions."""
    N, n_v, d, M = case["N"], case["n_v"], case["d"], case["M"]
    S, Q = case.get("S", S_SYS), case.get("Q", Q_IDS)
    gen = _gen(seed, 1)
    X = _randn(gen, N, n_v, d, dtype=torch.float32 if case["f32"] else torch.bfloat16)
    dirs = _randn(gen, max(M, 1) + 1, d)
    dirs /= dirs.norm(dim=1, keepdim=True)
    g, h = dirs[0], dirs[1:]
    order = torch.randperm(N, generator=gen, device=DEV)
    n_p, n_d = max(1, round(PLANTED * N)), round(DISTRACTORS * N)
    weak = torch.rand(max(n_d, 1), generator=gen, device=DEV)
    for k, i in enumerate(order[:n_p + n_d].tolist()):
        b = min(n_v, 16 + (7 * k) % 49)
        r0 = (13 * k) % max(1, n_v - b + 1)
        add = 8.0 * g if k < n_p else 8.0 * (0.3 + 0.4 * weak[k - n_p]) * g + 8.0 * h[0]
        X[i, r0:r0 + b] += add.to(X.dtype)
    vocab = 2000
    E = _randn(gen, vocab, d, scale=0.02)
    ids = torch.randperm(vocab, generator=gen, device=DEV)[:S + Q + max(M, 1)].to(torch.int32)
    sys_ids, q_ids, bg_ids = ids[:S].contiguous(), ids[S:S + Q].contiguous(), ids[S + Q:].contiguous()
    beta = 0.02 * math.sqrt(d)
    E[q_ids.long()] += beta * g
    E[bg_ids.long()] += beta * h
    return SimpleNamespace(X=X, embed=E.to(torch.bfloat16), sys=sys_ids, q=q_ids, bg=bg_ids, S=S, Q=Q)


def _decoder(case):
    hd = case["d"] // case["heads"]
    return SimpleNamespace(n_layers=case["layers"], d=case["d"], n_heads=case["heads"], head_dim=hd, ffn=case["ffn"],
                           vocab=case["vocab"], eps=1e-6, rope_theta=1e4)


def _weights(case, seed):
    """Random-init decoder weights: projections N(0, 0.02) in fp16, gains 1 + 0.1 N(0, 1) in bf16."""
    d, f = case["d"], case["ffn"]
    shapes = dict(wq=(d, d), wk=(d, d), wv=(d, d), wo=(d, d), wg=(f, d), wu=(f, d), wd=(d, f))
    layers = []
    for l in range(case["layers"]):
        gen = _gen(seed, 2, l)
        W = {k: _randn(gen, *s, dtype=torch.float16, scale=0.02) for k, s in shapes.items()}
        for k in ("g_attn", "g_ffn"):
            W[k] = (1.0 + 0.1 * _randn(gen, d)).to(torch.bfloat16)
        layers.append(W)
    gen = _gen(seed, 3)
    g_final = (1.0 + 0.1 * _randn(gen, d)).to(torch.bfloat16)
    lm = _randn(gen, case["vocab"], d, dtype=torch.float16, scale=0.02)
    return layers, g_final, lm


def _lengths(case, prompt=S_SYS + Q_IDS):
    """Sequence lengths of kept tiles: prompt rows plus a budget each.  mix 0: the smallest budget;
    1: the 400-tile scene's mix (seven of eight at 288, the rest 144 and 72); 2: the full tile."""
    out = []
    for i in range(case["seqs"]):
        if case["mix"] == 0:
            b = 72
        elif case["mix"] == 2:
            b = 576
        else:
            b = 144 if i % 8 == 3 else 72 if i % 24 == 7 else 288
        out.append(prompt + b + (case["extra"] * (i + 1)) % 41)
    return out


def _offsets(lengths):
    cu = [0]
    for n in lengths:
        cu.append(cu[-1] + n)
    pos = torch.cat([torch.arange(n, dtype=torch.int32, device=DEV) for n in lengths])
    return torch.tensor(cu, dtype=torch.int32, device=DEV), pos, cu


def _attn_lengths(case):
    L = case["L"]
    return [max(1, L - (37 * i) % max(1, L // 2)) if case["ragged"] else L for i in range(case["seqs"])]


def _pipeline(case, sc, policy, model=None):
    pipe = ScenePipeline(case["N"], case["n_v"], case["d"], "f32" if case["f32"] else "bf16", case["M"], sc.S, sc.Q,
                         case["knn"], policy, model=model, device=DEV)
    # what lies past a buffer's count is never written: give it a value
    for t in (pipe.nbr, pipe.u, pipe.kept, pipe.budgets, pipe.sel, pipe.sel_off, pipe.packed, pipe.positions, pipe.cu,
              pipe.ctx, pipe.ctx_off, pipe.ctx_target):
        if t is not None:
            t.zero_()
    return pipe


def prepare(case, seed):
    kind = case["kind"]
    st = SimpleNamespace(case=case, kind=kind)
    if kind in ("scene", "features", "query"):
        sc = st.sc = _scene(case, seed)
        if kind == "query":
            layers, g_final, lm = _weights(case, seed)
            st.model = DeviceModel(_decoder(case), layers, g_final, DEV, lm_head=lm)
            del layers
            st.logits = torch.zeros(case["N"], case["vocab"], dtype=torch.float32, device=DEV)
        st.pipe = _pipeline(case, sc, _policy(case), st.model if kind == "query" else None)
        if kind == "features":  # a selected scene is what the features are computed on
            st.n_kept, _ = st.pipe.run(sc.X, sc.embed, sc.q, sc.bg, sc.sys, sc.q, prefill=False)
            st.features = torch.zeros(case["N"], abi.N_FEATURES, dtype=torch.float32, device=DEV)
            st.V = torch.zeros(case["N"], case["d"], dtype=torch.float32, device=DEV)
            st.need = abi.features_workspace_bytes(case["N"], case["d"])
            st.ws = torch.empty(st.need, dtype=torch.uint8, device=DEV)
        return st
    if kind == "attention":
        cu, _, host = _offsets(_attn_lengths(case))
        st.T, st.cu, st.n, d = host[-1], cu, case["seqs"], case["heads"] * case["hd"]
        st.qkv = _randn(_gen(seed, 4), st.T, 3 * d, dtype=torch.float16)
        st.out = torch.empty(st.T, d, dtype=torch.float16, device=DEV)
        st.need = abi.attention_workspace_bytes(st.T, st.n)
        st.ws = torch.empty(max(st.need, 256), dtype=torch.uint8, device=DEV)
        return st
    layers, g_final, lm = _weights(case, seed)
    st.model = DeviceModel(_decoder(case), layers, g_final, DEV, lm_head=lm)
    del layers, lm
    d, L = case["d"], case["layers"]
    prompt = Q_IDS if kind == "prefix" else S_SYS + Q_IDS
    lengths = _lengths(case, prompt)
    st.cu, st.pos, host = _offsets(lengths)
    st.T, st.n = host[-1], case["seqs"]
    gen = _gen(seed, 5)
    st.logits = torch.empty(st.n, case["vocab"], dtype=torch.float32, device=DEV)
    if kind == "decode":
        st.max_len = max(lengths) + 1
        st.kv = _randn(gen, L, 2, st.T, d, dtype=torch.float16)
        st.embed = _randn(gen, 2000, d, dtype=torch.bfloat16)
        st.ids = torch.randint(0, 2000, (st.n,), dtype=torch.int32, device=DEV, generator=gen)
        st.hidden = torch.empty(st.n, d, dtype=torch.bfloat16, device=DEV)
        st.kv_new = torch.empty(L, 2, st.n, d, dtype=torch.float16, device=DEV)
        st.need = abi.decode_workspace_bytes(st.model.struct, st.n, st.max_len)
    else:
        st.rows = _randn(gen, st.T, d, dtype=torch.bfloat16)
        st.hidden = torch.empty_like(st.rows)
        if kind == "prefill":
            st.max_len = max(lengths)
            st.kv = torch.empty(L, 2, st.T, d, dtype=torch.float16, device=DEV)
            st.need = abi.prefill_workspace_bytes(st.model.struct, st.T, st.n, st.max_len)
        else:
            S = case["S"]
            st.max_len = S + max(lengths)
            st.embed = _randn(gen, 500, d, dtype=torch.bfloat16)
            st.sys = torch.randint(0, 500, (S,), dtype=torch.int32, device=DEV, generator=gen)
            st.prefix_hidden = torch.empty(S, d, dtype=torch.bfloat16, device=DEV)
            st.prefix_kv = torch.empty(L, 2, S, d, dtype=torch.float16, device=DEV)
            st.need = abi.prefill_shared_prefix_workspace_bytes(st.model.struct, st.T, st.n, st.max_len, S)
    st.ws = torch.empty(st.need, dtype=torch.uint8, device=DEV)
    return st


# ---------------------------------------------------------------------------------------- one pass

def run(st):
    kind, case = st.kind, st.case
    if kind == "scene":
        p, sc = st.pipe, st.sc
        p.run(sc.X, sc.embed, sc.q, sc.bg, sc.sys, sc.q, prefill=False, counts=False)
        out = dict(token_scores=p.token_scores, tile_s_raw=p.tile_s_raw, tile_s=p.tile_s, nbr=p.nbr, u=p.u, kept=p.kept,
                   n_kept=p.n_kept, budgets=p.budgets, sel=p.sel, sel_off=p.sel_off, packed=p.packed, cu=p.cu,
                   positions=p.positions, T=p.T)
        if case["merge"]:
            out.update(ctx_off=p.ctx_off, ctx_target=p.ctx_target, ctx=p.ctx)
        return out
    if kind == "features":
        p = st.pipe
        abi.tile_features(st.sc.X, p.xdt, p.N, p.n_v, p.d, p.t, p.B if p.M else None, p.M, p.token_scores, p.kept,
                          p.n_kept, st.features, st.V, st.ws, st.need)
        return dict(features=st.features, V=st.V)
    if kind == "query":
        p, sc = st.pipe, st.sc
        p.select(sc.X, sc.embed, sc.q, sc.bg)
        p.pack(sc.X, sc.embed, sc.sys, sc.q)
        p.prefill(last_logits=st.logits)
        return dict(n_kept=p.n_kept, budgets=p.budgets, sel_off=p.sel_off, T=p.T, hidden=p.packed, logits=st.logits)
    if kind == "attention":
        abi.attention_varlen(st.qkv, st.T, st.cu, st.n, case["heads"], case["hd"], st.out, st.ws, st.need)
        return st.out
    m = st.model.struct
    if kind == "decode":
        abi.decode_step(m, st.kv, st.T, st.cu, st.n, st.max_len, st.ids, st.embed, 2000, st.hidden, st.kv_new,
                        st.logits, st.ws, st.need)
        return dict(hidden=st.hidden, kv_new=st.kv_new, logits=st.logits)
    st.hidden.copy_(st.rows)  # the prefill works in place on the packed rows
    if kind == "prefill":
        abi.prefill_layers(m, st.hidden, st.T, st.cu, st.n, st.max_len, st.pos, st.ws, st.need, kv_out=st.kv,
                           last_logits=st.logits)
        return dict(hidden=st.hidden, kv=st.kv, logits=st.logits)
    abi.prefill_shared_prefix(m, st.sys, case["S"], st.embed, 500, st.prefix_hidden, st.prefix_kv, st.hidden, st.T,
                              st.cu, st.n, st.max_len, st.pos, st.logits, st.ws, st.need)
    return dict(hidden=st.hidden, prefix_hidden=st.prefix_hidden, prefix_kv=st.prefix_kv, logits=st.logits)


# ---------------------------------------------------------------------------------------- cost and tolerance

def _layer_work(case, rows, lengths, S=0):
    d, f, L = case["d"], case["ffn"], case["layers"]
    per = 4 * d * d + 3 * d * f
    attn = sum(4 * d * (n * (n + 1) / 2 + n * S) for n in lengths)
    return L * per * 2, L * (2 * rows * per + attn)  # weight bytes, flops


def _query_counts(case):
    n = max(1, round(KEPT * case["N"]))
    b = MEAN_BUDGET * case["n_v"]
    return n, b, case.get("S", 0) + case.get("Q", 0)


def work(case):
    kind = case["kind"]
    if kind in ("scene", "query"):
        N, n_v, d = case["N"], case["n_v"], case["d"]
        e = 4 if case["f32"] else 2
        n, b, prompt = _query_counts(case)
        rows = n * (b + prompt)
        # every token read once, the scores written, the packed rows written (the selected tokens'
        # second read and, with the merge, the kept tiles' are not needed a third time)
        byts = N * n_v * (d * e + 4) + n * b * d * e + rows * d * 2
        flops = 4.0 * N * n_v * d + 2.0 * N * N * d
        if case.get("merge"):
            m = 10 * b / 64
            byts += n * (n_v - b) * d * e
            flops += 2.0 * n * (n_v - b) * m * d
        if kind == "query":
            wb, fl = _layer_work(case, rows, [b + prompt] * n)
            byts += wb + case["vocab"] * d * 2 + n * case["vocab"] * 4
            flops += fl + 2.0 * n * d * case["vocab"]
        return dict(bytes=byts, flops=flops)
    if kind == "features":
        n = max(1, round(KEPT * case["N"]))
        e = 4 if case["f32"] else 2
        return dict(bytes=n * case["n_v"] * (case["d"] * e + 4) + n * case["d"] * 4,
                    flops=float(n * case["n_v"] * case["d"]))
    if kind == "attention":
        d, ls = case["heads"] * case["hd"], _attn_lengths(case)
        return dict(bytes=8 * d * sum(ls), flops=float(sum(2 * d * n * (n + 1) for n in ls)))
    ls = _lengths(case, Q_IDS if kind == "prefix" else S_SYS + Q_IDS)
    T, n, d, L, V = sum(ls), case["seqs"], case["d"], case["layers"], case["vocab"]
    head = (V * d * 2 + n * V * 4, 2.0 * n * d * V)
    if kind == "decode":
        wb, fl = _layer_work(case, n, [])
        return dict(bytes=wb + head[0] + L * 2 * (T + n) * d * 2 + n * d * 4, flops=fl + head[1] + L * 4.0 * d * (T + n))
    if kind == "prefill":
        wb, fl = _layer_work(case, T, ls)
        return dict(bytes=wb + head[0] + T * d * 4 + L * 2 * T * d * 2, flops=fl + head[1])
    S = case["S"]
    wb, fl = _layer_work(case, T, ls, S)
    _, fp = _layer_work(case, S, [S])
    return dict(bytes=wb + head[0] + (T + S) * d * 4 + L * 2 * S * d * 2, flops=fl + fp + head[1])


def tolerance(case):
    kind = case["kind"]
    if kind in ("scene", "features"):
        # 32-bit sums over up to 4096 terms; ties between scores that close may fall the other way
        return {"rel": 1e-5, "max": 1e-3, "differ": 0.005}
    if kind == "attention":
        return {"rel": 1e-3, "max": 0.05}  # fp16 weights and output
    if kind == "query":
        return {"rel": 0.01, "max": 0.3, "differ": 0.005}  # 32 layers of fp16 operands
    return {"rel": 6e-3, "max": 0.1}  # a few layers of fp16 operands, bf16 hidden states


# ---------------------------------------------------------------------------------------- 64 bits

F64 = torch.float64


def _norm(x):
    return x / x.norm(dim=-1, keepdim=True)


def _rms(x, g, eps=1e-6):
    return x / torch.sqrt((x * x).mean(dim=-1, keepdim=True) + eps) * g.to(F64)


def _rope(x, pos, theta=1e4):
    """x [rows, heads, hd], rotate-half pairs (j, j + hd / 2)."""
    hd = x.shape[-1]
    inv = theta ** (-torch.arange(0, hd, 2, dtype=F64, device=DEV) / hd)
    ang = pos.to(F64)[:, None] * inv
    c, s = ang.cos()[:, None], ang.sin()[:, None]
    a, b = x[..., :hd // 2], x[..., hd // 2:]
    return torch.cat([a * c - b * s, b * c + a * s], dim=-1)


def _attend(q, k, v, offset):
    """Causal attention of rows offset .. offset + n - 1 over k, v (all rows up to each), per head."""
    n, H, hd = q.shape
    out = torch.empty_like(q)
    mask = torch.arange(k.shape[0], device=DEV)[None] > (torch.arange(n, device=DEV) + offset)[:, None]
    for h in range(H):
        s = (q[:, h] @ k[:, h].T) / math.sqrt(hd)
        out[:, h] = torch.softmax(s.masked_fill(mask, -math.inf), dim=-1) @ v[:, h]
    return out


def _layers64(case, seed, h, pos, attend):
    """The decoder over rows h: attend(layer, q, k, v) gives the attention output.  Returns the final
    hidden states and each layer's keys and values."""
    layers, g_final, lm = _weights(case, seed)
    H, d = case["heads"], case["d"]
    kv = []
    for l, W in enumerate(layers):
        x = _rms(h, W["g_attn"])
        q, k, v = ((x @ W[n].to(F64).T).view(-1, H, d // H) for n in ("wq", "wk", "wv"))
        q, k = _rope(q, pos), _rope(k, pos)
        kv.append(torch.stack([k.reshape(-1, d), v.reshape(-1, d)]))
        h = h + attend(l, q, k, v).reshape(-1, d) @ W["wo"].to(F64).T
        x = _rms(h, W["g_ffn"])
        g = x @ W["wg"].to(F64).T
        h = h + (g * torch.sigmoid(g) * (x @ W["wu"].to(F64).T)) @ W["wd"].to(F64).T
    return _rms(h, g_final), torch.stack(kv), lm.to(F64)


def _packed_attend(cu, H, hd, prefix=None):
    def attend(l, q, k, v):
        out = torch.empty_like(q)
        for a, b in zip(cu[:-1], cu[1:]):
            kk, vv, S = k[a:b], v[a:b], 0
            if prefix is not None:
                S = prefix.shape[2]
                kk = torch.cat([prefix[l, 0].view(S, H, hd), kk])
                vv = torch.cat([prefix[l, 1].view(S, H, hd), vv])
            out[a:b] = _attend(q[a:b], kk, vv, S)
        return out
    return attend


def _scores64(case, seed):
    sc = _scene(case, seed)
    N, M, m = case["N"], case["M"], min(case["knn"], case["N"] - 1)
    t = _norm(sc.embed[sc.q.long()].to(F64).mean(dim=0))
    w = t - _norm(sc.embed[sc.bg.long()].to(F64)).mean(dim=0) if M else t
    r, V = [], []
    for i in range(N):
        x = sc.X[i].to(F64)
        r.append(x @ w / x.norm(dim=1))
        V.append(_norm(x.sum(dim=0)))
    V = torch.stack(V)
    s = V @ w
    st = s
    if m > 0:
        G = V @ V.T
        G.fill_diagonal_(-math.inf)
        st = (s + s[G.topk(m, dim=1).indices].sum(dim=1)) / (m + 1)
    span = st.max() - st.min()
    u = (st - st.min()) / span if float(span) > 1e-12 else None
    return sc, w, torch.stack(r), V, s, st, u


def exact(case, seed):
    kind = case["kind"]
    if kind == "query":
        return None
    if kind == "scene":
        _, _, r, _, s, st, u = _scores64(case, seed)
        names = ["nbr", "kept", "n_kept", "budgets", "sel", "sel_off", "packed", "cu", "positions", "T"]
        names += ["ctx_off", "ctx_target", "ctx"] if case["merge"] else []
        # with every tile in each other's neighbourhood the smoothed scores are all the same number,
        # and u is decided by how it is rounded
        return dict(token_scores=r, tile_s_raw=s, tile_s=st, u=None if case["knn"] >= case["N"] - 1 else u,
                    **{k: None for k in names})
    if kind == "features":
        st = prepare(case, seed)
        sc, w, r, V, _, _, _ = _scores64(case, seed)
        g = math.isqrt(case["n_v"])
        kept = st.pipe.kept[:st.n_kept].long()
        f = torch.zeros(case["N"], abi.N_FEATURES, dtype=F64, device=DEV)
        Vk = torch.zeros(case["N"], case["d"], dtype=F64, device=DEV)
        for j, i in enumerate(kept.tolist()):
            x = sc.X[i].to(F64).view(2, g // 2, 2, g // 2, -1).sum(dim=(1, 3)).view(4, -1)
            f[j] = torch.cat([_norm(x) @ w, r[i].max()[None], r[i].mean()[None], r[i].std(unbiased=False)[None]])
            Vk[j] = V[i]
        return dict(features=f, V=Vk)
    st = prepare(case, seed)
    if kind == "attention":
        H, hd = case["heads"], case["hd"]
        q, k, v = (x.to(F64).view(-1, H, hd) for x in st.qkv.view(st.T, 3, H * hd).unbind(1))
        return _packed_attend(st.cu.tolist(), H, hd)(0, q, k, v).view(st.T, H * hd)
    H, d, cu = case["heads"], case["d"], st.cu.tolist()
    hd = d // H
    if kind == "decode":
        lens = [b - a for a, b in zip(cu[:-1], cu[1:])]

        def attend(l, q, k, v):
            out = torch.empty_like(q)
            for i, (a, b) in enumerate(zip(cu[:-1], cu[1:])):
                kk = torch.cat([st.kv[l, 0, a:b].to(F64).view(-1, H, hd), k[i:i + 1]])
                vv = torch.cat([st.kv[l, 1, a:b].to(F64).view(-1, H, hd), v[i:i + 1]])
                p = torch.softmax(torch.einsum("hd,khd->hk", q[i], kk) / math.sqrt(hd), dim=-1)
                out[i] = torch.einsum("hk,khd->hd", p, vv)
            return out

        pos = torch.tensor(lens, device=DEV)
        h, kv, lm = _layers64(case, seed, st.embed[st.ids.long()].to(F64), pos, attend)
        return dict(hidden=h, kv_new=kv, logits=h @ lm.T)
    prefix, S = None, 0
    if kind == "prefix":
        S = case["S"]
        ph, prefix, _ = _layers64(case, seed, st.embed[st.sys.long()].to(F64), torch.arange(S, device=DEV),
                                  _packed_attend([0, S], H, hd))
    h, kv, lm = _layers64(case, seed, st.rows.to(F64), st.pos + S, _packed_attend(cu, H, hd, prefix))
    logits = h[torch.tensor(cu[1:], device=DEV) - 1] @ lm.T
    if kind == "prefix":
        return dict(hidden=h, prefix_hidden=ph, prefix_kv=prefix, logits=logits)
    return dict(hidden=h, kv=kv, logits=logits)
