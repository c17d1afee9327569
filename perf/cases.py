"""Performance cases of the VoxZip path: what a serving program calls, over the sizes it meets.

A request runs stage 1 once (on the prefilled K/V, or on the input embeddings), then one decode
step per generated token and an eviction every 32 steps. The cases are those calls, through the
package's public entry points, from one 1-layer fp32 step to an hour of audio for four sequences.

kind "decode"   one or more decode steps. launch "eager": one call for all layers, from the host;
                "layers": a CUDA graph of one call per layer and step, as a model issues them (the
                queries of a layer need the layer below); "steps": a CUDA graph of one call per
                step for all layers. Each pass first drops the tokens the last one appended (a
                program that rejects drafted tokens, or answers again), by copying the lengths back.
kind "evict"    one eviction of all layers. Each pass first copies back the scores, positions and
                lengths as the interval's decode steps left them; the rows need no copy, since
                what the eviction does depends on the scores and positions alone.
kind "fuse"     stage 1 on the prefilled K/V of every layer.
kind "embed"    stage 1 on the input embeddings, from ASR segments.
kind "request"  stage 1 and the first steps of the reply through Session, the decode loop replayed
                from its CUDA graph. It ends before the first eviction: which row an eviction
                drops may hang on the last bit of a score, and what follows would then differ.

Lengths, spans and segments belong to the case ("layout" seeds them); values come from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_08569_gb300 import (PAGE_TOKENS, CacheDesc, EmbedDesc, allocate_paged_cache, voxzip_anchor_fuse,
                                    voxzip_anchor_fuse_workspace_size, voxzip_decode_step, voxzip_decode_step_paged,
                                    voxzip_embed_fuse, voxzip_embed_fuse_workspace_size, voxzip_evict,
                                    voxzip_evict_ex, voxzip_get_status, voxzip_segments_to_spans)
from paper_2608_08569_gb300 import workloads as W
from paper_2608_08569_gb300.session import Session

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
THINKER = dict(layers=48, q_heads=32, kv_heads=4, head_dim=128, dtype="bf16")


# ----------------------------------------------------------------------------- the cases

def _decode(name, *, batch, n, launch, steps=1, ragged=False, paged=False, gamma=0.99, layout=0, **shape):
    return dict(name=name, kind="decode", batch=batch, n=n, launch=launch, steps=steps, ragged=ragged, paged=paged,
                gamma=gamma, layout=layout, **shape)


def _evict(name, *, batch, budget, n, compaction="ordered", history=True, layout=0, **shape):
    return dict(name=name, kind="evict", batch=batch, budget=budget, n=n, compaction=compaction, history=history,
                layout=layout, **shape)


def listed():
    return [
        # The smallest call: one fp32 layer, 150 cached rows, issued from the host.
        _decode("decode_tiny_f32", batch=1, n=149, launch="eager", gamma=0.95, layers=1, q_heads=2, kv_heads=1,
                head_dim=64, dtype="f32"),
        # An fp32 cache of the full shape: 10 min of audio at a 20x budget, one call from the host.
        _decode("decode_f32_10min", batch=1, n=416, launch="eager", **dict(THINKER, dtype="f32")),
        # One token of a 10-min request at 20x, layer by layer as the model runs it.
        _decode("token_10min", batch=1, n=416, launch="layers", **THINKER),
        # One token of 32 ragged sequences of 2-8 min at 4x, layer by layer.
        _decode("token_batch32", batch=32, n=1564, launch="layers", ragged=True, gamma=0.98, layout=4, **THINKER),
        # Tokens of four 60-min requests at 20x, one call per token.
        _decode("decode_60min", batch=4, n=2317, launch="steps", steps=4, gamma=0.995, **THINKER),
        # Tokens of a 10-min request at 4x on a paged cache.
        _decode("decode_paged_10min", batch=1, n=2019, launch="steps", steps=4, paged=True, **THINKER),
        # The eviction after 32 tokens: a 30-s clip at 4x, and four 60-min requests at 20x.
        _evict("evict_30s", batch=1, budget=157, n=189, **THINKER),
        _evict("evict_60min", batch=4, budget=2301, n=2333, **THINKER),
        # The same with hole filling, which moves only the rows beyond the budget.
        _evict("evict_fill_60min", batch=4, budget=2301, n=2333, compaction="fill", **THINKER),
        # Stage 1 of four 60-min prompts, on K/V (5% silences) and on embeddings.
        dict(name="fuse_60min", kind="fuse", batch=4, audio=45000, text=1024, ragged=False, span_mean=6.0,
             silence=0.05, anchors=False, layout=5, **THINKER),
        dict(name="embed_60min", kind="embed", batch=4, audio=45000, text=1024, ragged=False, d_model=2048,
             dtype="bf16", anchors=True, keep_background=True, layout=12),
        # A 30-s clip from its prefilled prompt to the last token before the first eviction.
        dict(name="request_30s", kind="request", batch=1, audio=375, text=256, ragged=False, span_mean=4.0,
             silence=0.0, steps=31, gamma=0.98, layout=1, **THINKER),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_shape(rng, f32):
    r = rng.random()
    if r < 0.7:
        return dict(THINKER, dtype="f32" if f32 else "bf16")
    heads, kv, dim = rng.choice([(16, 1, 64), (12, 3, 128), (4, 4, 128), (2, 1, 64), (32, 8, 128)])
    return dict(layers=_log(rng, 1, 48), q_heads=heads, kv_heads=kv, head_dim=dim, dtype="f32" if f32 else "bf16")


def _draw_once(rng):
    kind = rng.choice(["decode", "decode", "decode", "evict", "evict", "fuse", "embed", "request"])
    batch, audio, text = _log(rng, 1, 32), _log(rng, 375, 45000), _log(rng, 32, 1024)
    budget = max(16, (audio + text) // rng.choice([4, 20]))
    layout = rng.randrange(1 << 20)
    f32 = rng.random() < 0.2
    if kind == "decode":
        launch = rng.choice(["eager", "layers", "steps"])
        paged = not f32 and rng.random() < 0.25
        return _decode("", batch=batch, n=budget + rng.randrange(32), launch=launch,
                       steps=rng.randrange(2, 5) if launch == "steps" else 1, ragged=batch > 1 and rng.random() < 0.5,
                       paged=paged, gamma=rng.choice([0.95, 0.98, 0.99, 0.995, 1.0]), layout=layout,
                       **_draw_shape(rng, f32))
    if kind == "evict":
        return _evict("", batch=batch, budget=budget, n=budget + rng.choice([16, 32, 32, 32, 3 * budget]),
                      compaction=rng.choice(["ordered", "ordered", "fill"]), history=rng.random() < 0.85,
                      layout=layout, **_draw_shape(rng, f32))
    ragged = batch > 1 and rng.random() < 0.5
    if kind == "embed":
        return dict(kind="embed", batch=batch, audio=audio, text=text, ragged=ragged,
                    d_model=rng.choice([64, 256, 1000, 2048]), dtype="f32" if f32 else "bf16",
                    anchors=rng.random() < 0.7, keep_background=rng.random() < 0.7, layout=layout)
    spans = dict(span_mean=rng.choice([4.0, 5.0, 6.0]), silence=rng.choice([0.0, 0.05]))
    if kind == "fuse":
        return dict(kind="fuse", batch=batch, audio=audio, text=text, ragged=ragged, anchors=rng.random() < 0.25,
                    layout=layout, **spans, **_draw_shape(rng, f32))
    return dict(kind="request", batch=batch, audio=audio, text=text, ragged=ragged, steps=rng.randrange(1, 32),
                gamma=rng.choice([0.98, 0.99, 0.995]), layout=layout, **spans, **_draw_shape(rng, f32))


def draw(rng):
    most = {k: max(work(c)["bytes"] for c in listed() if c["kind"] == k) for k in ("decode", "evict", "fuse", "embed")}
    most["request"] = most["fuse"] / 4
    while True:
        c = _draw_once(rng)
        if work(c)["bytes"] <= most[c["kind"]]:
            c.pop("name", None)
            return c


# ----------------------------------------------------------------------------- sizes of a case

def _lens(c):
    """Rows of every sequence before the step (paged: no append of the pass starts a page)."""
    if c["ragged"]:
        lens = np.random.default_rng(c["layout"]).integers(-(-c["n"] // 4), c["n"] + 1, c["batch"])
        lens[0] = c["n"]
    else:
        lens = np.full(c["batch"], c["n"])
    if c["paged"]:
        lens = lens - np.maximum(0, lens % PAGE_TOKENS + c["steps"] - (PAGE_TOKENS - 1))
    return [max(0, int(x)) for x in lens]


def _audio(c):
    if not c["ragged"]:
        return (c["audio"],) * c["batch"]
    a = np.random.default_rng(c["layout"]).integers(-(-c["audio"] // 4), c["audio"] + 1, c["batch"])
    a[0] = c["audio"]
    return tuple(int(x) for x in a)


def _workload(c):
    return W.Workload("case", layers=c["layers"], q_heads=c["q_heads"], kv_heads=c["kv_heads"],
                      head_dim=c["head_dim"], dtype=DTYPES[c["dtype"]], batch=c["batch"], audio_len=_audio(c),
                      text_len=c["text"], budget=(c["audio"],) * c["batch"], gamma=c.get("gamma", 1.0),
                      steps=c.get("steps", 1), interval=32, span_mean=c["span_mean"], silence_prob=c["silence"],
                      seed=c["layout"])


def _embed_workload(c):
    return W.EmbedWorkload("case", batch=c["batch"], audio_len=_audio(c), text_len=c["text"], d_model=c["d_model"],
                           dtype=DTYPES[c["dtype"]], seed=c["layout"])


def _embed_spans(w):
    """CSR spans of the kept segments, from their times (Eq. 3)."""
    off, start, end, groups = [0], [], [], []
    for b, s in enumerate(W.make_segments(w)):
        r = voxzip_segments_to_spans(s.t_start, s.t_end, s.confidence, s.text_len, s.tau_total, w.audio_len[b],
                                     w.audio_begin)
        start += list(r["start"])
        end += list(r["end"])
        groups += list(r["groups"])
        off.append(len(start))
    a = lambda x: np.asarray(x, np.int32)
    return W.Spans(a(off), a(start), a(end), a(groups))


def _slots(w, spans, b, keep_background=True):
    """Output row of every prompt token of sequence b (-1: dropped), written out token by token as
    the definition has it, and the anchor row of every output row (-1: none)."""
    n = w.in_len[b]
    start, end, groups = spans.of(b)
    slot, anchors, row, anchor, t = np.full(n, -1, np.int64), [], 0, 0, 0
    audio_end = w.audio_begin + w.audio_len[b]

    def copied(upto):
        nonlocal t, row
        x = np.arange(t, upto)
        kept = x if keep_background else x[(x < w.audio_begin) | (x >= audio_end)]
        slot[kept] = row + np.arange(len(kept))
        anchors.extend([-1] * len(kept))
        row += len(kept)
        t = upto

    for s, e, ng in zip(start.tolist(), end.tolist(), groups.tolist()):
        copied(s)
        g = min(ng, e - s)
        cuts = [s + j * (e - s) // g for j in range(g + 1)] if g else []
        for j in range(g):
            slot[cuts[j]:cuts[j + 1]] = row + j
        anchors.extend(range(anchor, anchor + g))
        row += g
        anchor += ng
        t = e
    copied(n)
    return slot, np.asarray(anchors, np.int64), row


def _rows(w, spans, keep_background=True):
    """Stage-1 rows of every sequence."""
    out = []
    for b in range(w.batch):
        s, e, g = (x.astype(np.int64) for x in spans.of(b))
        dropped = 0 if keep_background else w.audio_len[b] - int((e - s).sum())
        out.append(int(w.in_len[b] + (np.minimum(g, e - s) - (e - s)).sum() - dropped))
    return out


def _size(c):
    return 2 if c["dtype"] == "bf16" else 4


def _decode_work(c, lens, steps):
    D, G, units, e = c["head_dim"], c["q_heads"] // c["kv_heads"], c["layers"] * c["kv_heads"], _size(c)
    rows = sum(n + t + 1 for n in lens for t in range(steps))
    fixed = (2 * G * D + 4 * D) * e + 4
    return units * (rows * (2 * D * e + 8) + len(lens) * steps * fixed), units * rows * 4 * G * D


def work(case):
    c = case
    e = _size(c)
    if c["kind"] == "decode":
        by, fl = _decode_work(c, _lens(c), c["steps"])
    elif c["kind"] == "evict":
        units, D = c["batch"] * c["layers"] * c["kv_heads"], c["head_dim"]
        m = int(0.2 * c["budget"])
        gone, hist = c["n"] - c["budget"], c["n"] - m - 4
        if not c["history"]:
            first = 4  # everything between the sinks and the recent window leaves
        else:  # the expected first of `gone` rows drawn among the history
            first = 4 + (hist - gone) // (gone + 1)
        moved = min(gone, c["budget"]) if c["compaction"] == "fill" else max(0, c["budget"] - first)
        by, fl = units * (8 * c["n"] + 2 * (2 * D * e + 8) * moved), 0
    elif c["kind"] == "embed":
        w = _embed_workload(c)
        spans = _embed_spans(w)
        rows = sum(_rows(w, spans, c["keep_background"]))
        text = int(np.minimum(spans.groups, spans.end - spans.start).sum()) if c["anchors"] else 0
        read = sum(w.in_len) if c["keep_background"] else sum(w.in_len) - sum(w.audio_len) + int((spans.end - spans.start).sum())
        by, fl = (read + rows + text) * c["d_model"] * e + 4 * rows, read * c["d_model"]
    else:
        w = _workload(c)
        spans = W.make_spans(w)
        rows, units, D = _rows(w, spans), c["layers"] * c["kv_heads"], c["head_dim"]
        anchor = 2 * len(spans.start) * D * e if c.get("anchors") else 0
        by = units * (2 * sum(w.in_len) * D * e + sum(rows) * (2 * D * e + 8) + anchor)
        fl = units * 2 * sum(w.in_len) * D
        if c["kind"] == "request":
            db, df = _decode_work(c, rows, c["steps"])
            by, fl = by + db, fl + df
    return {"bytes": int(by), "flops": int(fl)}


# ----------------------------------------------------------------------------- inputs

class State:
    """What one case has in hand; fields by kind."""


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(shape, dtype, g):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=g)


def _i32(x):
    return torch.as_tensor(np.asarray(x), dtype=torch.int32, device="cuda")


def _key_scale(c, rng):
    """[L][Hkv][D]: 4 outlier channels per layer and kv-head, x16."""
    s = np.ones((c["layers"], c["kv_heads"], c["head_dim"]), np.float32)
    for l in range(c["layers"]):
        for h in range(c["kv_heads"]):
            s[l, h, rng.choice(c["head_dim"], 4, replace=False)] = 16.0
    return torch.from_numpy(s).cuda()


def _step_inputs(c, steps, scale, g):
    """q [S][L][B][Hq][D] (half noise, half a mix of 8 directions per layer and kv-head), k_new and
    v_new [S][L][B][Hkv][D]."""
    L, B, Hq, H, D, dt = c["layers"], c["batch"], c["q_heads"], c["kv_heads"], c["head_dim"], DTYPES[c["dtype"]]
    dirs = _normal((L, H, 8, D), torch.float32, g)
    mix = _normal((steps, L, B, H, Hq // H, 8), torch.float32, g) / math.sqrt(8)
    q = 0.5 * _normal((steps, L, B, H, Hq // H, D), torch.float32, g)
    q += 0.5 * torch.einsum("slbhga,lhad->slbhgd", mix, dirs)
    kn = _normal((steps, L, B, H, D), torch.float32, g) * scale[None, :, None]
    return q.reshape(steps, L, B, Hq, D).to(dt), kn.to(dt), _normal((steps, L, B, H, D), dt, g)


def _fill_positions(pos, g):
    """Ascending positions with gaps of 1 to 7 tokens."""
    gaps = torch.randint(1, 8, pos.shape, generator=g, device="cuda", dtype=torch.int32)
    pos.copy_(gaps.cumsum(-1, dtype=torch.int32))


def _decode_step(s, t, l, count):
    """Step t of layers [l, l + count)."""
    q, kn, vn, out = (x[t, l:l + count] for x in (s.q, s.kn, s.vn, s.out))
    if s.paged:
        voxzip_decode_step_paged(s.desc, s.paged, l, count, q, kn, vn, s.new_pos[t], s.gamma, out, max_len=s.n + t + 1)
    else:
        voxzip_decode_step(s.desc, l, count, q, kn, vn, s.new_pos[t], s.k, s.v, s.score, s.pos, s.len, s.gamma, out,
                           max_len=s.n + t + 1)


def _prepare_decode(c, seed):
    s, g, dt = State(), _generator(seed), DTYPES[c["dtype"]]
    B, L, H, D, steps = c["batch"], c["layers"], c["kv_heads"], c["head_dim"], c["steps"]
    lens = _lens(c)
    capacity = max(lens) + steps + 32
    capacity = -(-capacity // PAGE_TOKENS) * PAGE_TOKENS if c["paged"] else capacity
    s.desc = desc = CacheDesc(B, L, c["q_heads"], H, D, capacity, dt)
    scale = _key_scale(c, np.random.default_rng(seed))
    k = _normal((B, L, H, capacity, D), dt, g).mul_(scale[None, :, :, None, :])
    v = _normal((B, L, H, capacity, D), dt, g)
    s.len0 = _i32(lens)[:, None, None].expand(B, L, H).contiguous()
    s.score = torch.empty(B, L, H, capacity, device="cuda")
    s.pos = torch.empty(B, L, H, capacity, dtype=torch.int32, device="cuda")
    _fill_positions(s.pos, g)
    if c["paged"]:  # every unit's pages, in an order of their own
        pages = B * L * H * (capacity // PAGE_TOKENS)
        order = torch.randperm(pages, generator=g, device="cuda")
        pc = allocate_paged_cache(desc, pages)
        pc["k_pool"][order] = k.view(pages, PAGE_TOKENS, D)
        pc["v_pool"][order] = v.view(pages, PAGE_TOKENS, D)
        pc["page_table"].copy_(order.view(pc["page_table"].shape))
        pc["free_count"].zero_()
        pc.update(score=s.score, pos=s.pos)
        s.paged, s.len, s.k, s.v = pc, pc["len"], pc["k_pool"], pc["v_pool"]
    else:
        s.paged, s.len, s.k, s.v = None, s.len0.clone(), k, v
    s.q, s.kn, s.vn = _step_inputs(c, steps, scale, g)
    s.new_pos = torch.stack([s.pos.amax() + 1 + t for t in range(steps)])[:, None].expand(steps, B).contiguous()
    s.out = torch.empty_like(s.q)
    s.gamma, s.steps, s.n, s.graph = c["gamma"], steps, max(lens), None

    if c["launch"] != "eager":
        s.score.zero_()
        s.len.copy_(s.len0)
        _decode_step(s, 0, 0, 1 if c["launch"] == "layers" else L)  # loads the kernels before the capture
        torch.cuda.synchronize()
        s.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.graph):
            s.len.copy_(s.len0)
            for t in range(steps):
                for l in range(L if c["launch"] == "layers" else 1):
                    _decode_step(s, t, l, 1 if c["launch"] == "layers" else L)
    # decayed sums of the softmax mass a step adds
    s.score.exponential_(1.0, generator=g).mul_(c["q_heads"] / H / (max(1, s.n) * (1.005 - c["gamma"])))
    s.len.copy_(s.len0)
    return s


def _prepare_evict(c, seed):
    s, g, dt = State(), _generator(seed), DTYPES[c["dtype"]]
    B, L, H, D = c["batch"], c["layers"], c["kv_heads"], c["head_dim"]
    capacity = c["n"] + 32
    s.desc = CacheDesc(B, L, c["q_heads"], H, D, capacity, dt)
    s.k = _normal((B, L, H, capacity, D), dt, g)
    s.v = _normal((B, L, H, capacity, D), dt, g)
    slots, units = B * L * H * capacity, B * L * H
    s.live = torch.empty(2 * slots + units, dtype=torch.int32, device="cuda")  # scores, positions and lengths
    s.score = s.live[:slots].view(torch.float32).view(B, L, H, capacity)
    s.pos = s.live[slots:2 * slots].view(B, L, H, capacity)
    s.len = s.live[2 * slots:].view(B, L, H)
    s.score.exponential_(1.0, generator=g)
    _fill_positions(s.pos, g)
    s.len.fill_(c["n"])
    s.before = s.live.clone()
    s.budget, s.rows = _i32([c["budget"]] * B), c["budget"]
    s.compaction, s.history = c["compaction"], c["history"]
    return s


def _prepare_fuse(c, seed):
    s, g, w = State(), _generator(seed), _workload(c)
    spans = W.make_spans(w)
    B, L, H, D, dt = w.batch, w.layers, w.kv_heads, w.head_dim, w.dtype
    s.w, s.spans = w, spans
    scale = _key_scale(c, np.random.default_rng(seed))
    s.k_pre = _normal((B, L, H, w.stride, D), dt, g).mul_(scale[None, :, :, None, :])
    s.v_pre = _normal((B, L, H, w.stride, D), dt, g)
    s.ints = (_i32(w.in_len), _i32([w.audio_begin] * B), _i32(w.audio_len), _i32(spans.off), _i32(spans.start),
              _i32(spans.end), _i32(spans.groups))
    s.anchor_k = s.anchor_v = None
    if c.get("anchors"):
        a = max(1, int(np.diff(spans.off).max()))
        s.anchor_k, s.anchor_v = (_normal((B, L, H, a, D), dt, g) for _ in range(2))
    rows = _rows(w, spans)
    s.desc = CacheDesc(B, L, w.q_heads, H, D, max(rows) + c.get("steps", 0) + 32, dt)
    s.cache = dict(k=torch.zeros(B, L, H, s.desc.capacity, D, dtype=dt, device="cuda"),
                   v=torch.zeros(B, L, H, s.desc.capacity, D, dtype=dt, device="cuda"),
                   score=torch.zeros(B, L, H, s.desc.capacity, device="cuda"),
                   pos=torch.zeros(B, L, H, s.desc.capacity, dtype=torch.int32, device="cuda"),
                   len=torch.zeros(B, L, H, dtype=torch.int32, device="cuda"))
    need = voxzip_anchor_fuse_workspace_size(s.desc, w.stride, len(spans.start))
    s.workspace = torch.empty(max(need, 256), dtype=torch.uint8, device="cuda")
    if c["kind"] == "request":
        s.session = Session(s.desc, w.budget, w.gamma, cache=s.cache)
        s.q, s.kn, s.vn = _step_inputs(c, c["steps"], scale, g)
        s.new_pos = _i32([[n + t for n in w.in_len] for t in range(c["steps"])])
        s.out = torch.empty_like(s.q)
        s.session.prefill(s.k_pre, s.v_pre, *s.ints)
        s.session.decode(s.q[0], s.kn[0], s.vn[0], s.new_pos[0], s.out[0])  # loads the kernels before the capture
        s.session.prefill(s.k_pre, s.v_pre, *s.ints)
        s.graph = s.session.capture_loop(s.q, s.kn, s.vn, s.new_pos, s.out, w.interval)
        s.cache["k"].zero_()
        s.cache["v"].zero_()
    return s


def _prepare_embed(c, seed):
    s, g, w = State(), _generator(seed), _embed_workload(c)
    spans = _embed_spans(w)
    s.w, s.spans = w, spans
    B, D = w.batch, w.d_model
    s.e_in = _normal((B, w.stride, D), w.dtype, g)
    s.ints = (_i32(w.in_len), _i32([w.audio_begin] * B), _i32(w.audio_len), _i32(spans.off), _i32(spans.start),
              _i32(spans.end), _i32(spans.groups))
    s.e_text = None
    if c["anchors"]:
        rows = max(1, max(int(spans.of(b)[2].sum()) for b in range(B)))
        s.e_text = _normal((B, rows, D), w.dtype, g).mul_(0.5)
    s.keep = c["keep_background"]
    s.desc = EmbedDesc(B, D, max(1, max(_rows(w, spans, s.keep))), w.dtype)
    s.e_out = torch.zeros(B, s.desc.capacity, D, dtype=w.dtype, device="cuda")
    s.pos = torch.zeros(B, s.desc.capacity, dtype=torch.int32, device="cuda")
    s.len = torch.zeros(B, dtype=torch.int32, device="cuda")
    need = voxzip_embed_fuse_workspace_size(s.desc, w.stride, len(spans.start))
    s.workspace = torch.empty(max(need, 256), dtype=torch.uint8, device="cuda")
    return s


def prepare(case, seed):
    make = {"decode": _prepare_decode, "evict": _prepare_evict, "fuse": _prepare_fuse, "request": _prepare_fuse,
            "embed": _prepare_embed}[case["kind"]]
    s = make(case, seed)
    s.kind = case["kind"]
    if voxzip_get_status() != 0:
        raise RuntimeError("the device status word is set")
    return s


# ----------------------------------------------------------------------------- one pass

def run(s):
    if s.kind == "decode":
        if s.graph is not None:
            s.graph.replay()
        else:
            s.len.copy_(s.len0)
            _decode_step(s, 0, 0, s.desc.layers)
        return dict(out=s.out, score=s.score, k=s.k, v=s.v, pos=s.pos, len=s.len)
    if s.kind == "evict":
        s.live.copy_(s.before)
        if s.history and s.compaction == "ordered":
            voxzip_evict(s.desc, 0, s.desc.layers, s.k, s.v, s.score, s.pos, s.len, s.budget)
        else:
            voxzip_evict_ex(s.desc, 0, s.desc.layers, s.k, s.v, s.score, s.pos, s.len, s.budget, history=s.history,
                            compaction=s.compaction)
        rows = lambda t: t[:, :, :, :s.rows]
        return dict(k=rows(s.k), v=rows(s.v), score=rows(s.score), pos=rows(s.pos), len=s.len)
    if s.kind == "embed":
        voxzip_embed_fuse(s.desc, s.e_in, *s.ints, s.e_out, s.pos, s.len, e_text=s.e_text, keep_background=s.keep,
                          workspace=s.workspace)
        return dict(e_out=s.e_out, pos=s.pos, len=s.len)
    k, v, score, pos, len_ = (s.cache[x] for x in ("k", "v", "score", "pos", "len"))
    if s.kind == "fuse":
        voxzip_anchor_fuse(s.desc, s.k_pre, s.v_pre, *s.ints, k, v, score, pos, len_, anchor_k=s.anchor_k,
                           anchor_v=s.anchor_v, workspace=s.workspace)
        return dict(k=k, v=v, score=score, pos=pos, len=len_)
    s.session.prefill(s.k_pre, s.v_pre, *s.ints)
    s.graph.replay()
    return dict(out=s.out, k=k, v=v, score=score, pos=pos, len=len_)


# ----------------------------------------------------------------------------- what it should give

def tolerance(case):
    # Evictions move rows and the header fixes stage 1's sums (fp32, in token order, one rounding),
    # so their bits are determined. Decoding: bf16 outputs, bf16 probabilities in P V; fp32 sums.
    if case["kind"] in ("evict", "fuse", "embed"):
        return "exact"
    return {"rel": 1e-2, "max": 0.05} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 1e-3}


def _exact_steps(q, kn, vn, k, v, score, lens, gamma):
    """Decode steps in 64 bits on k, v [B][L][H][C][D], score [B][L][H][C], lens [B]."""
    S, L, B, Hq, D = q.shape
    H, C = k.shape[2], k.shape[3]
    out = torch.empty(q.shape, dtype=torch.float64, device=q.device)
    final = torch.zeros(score.shape, dtype=torch.float64, device=q.device)
    slot = torch.arange(C, device=q.device)
    rows = torch.arange(B, device=q.device)
    for l in range(L):
        kl, vl, sl = k[:, l].double(), v[:, l].double(), score[:, l].double()
        for t in range(S):
            n = lens + t
            kl[rows, :, n] = kn[t, l].double()
            vl[rows, :, n] = vn[t, l].double()
            sl[rows, :, n] = 0.0
            ql = q[t, l].double().view(B, H, Hq // H, D)
            x = (ql @ kl.transpose(-1, -2)) / math.sqrt(D)
            x.masked_fill_((slot[None] > n[:, None])[:, None, None], -math.inf)
            p = torch.softmax(x, -1)
            out[t, l] = (p @ vl).reshape(B, Hq, D)
            live = (slot[None] <= n[:, None])[:, None]
            sl = torch.where(live, gamma * sl + p.sum(2), sl)
        final[:, l] = sl
    return out, final


def _exact_rows(x, w, spans, b, anchors, capacity, keep=True):
    """Stage-1 rows of sequence b in 64 bits: x [..., in_len, D] to [..., capacity, D]."""
    slot, anchor_of, n = _slots(w, spans, b, keep)
    kept = torch.as_tensor(np.nonzero(slot >= 0)[0], device=x.device)
    slot = torch.as_tensor(slot[slot >= 0], device=x.device)
    y = torch.zeros(x.shape[:-2] + (capacity, x.shape[-1]), dtype=torch.float64, device=x.device)
    y.index_add_(x.dim() - 2, slot, x[..., kept, :].double())
    y /= torch.bincount(slot, minlength=capacity).clamp(min=1)[:, None]
    if anchors is not None:
        rows = torch.as_tensor(np.nonzero(anchor_of >= 0)[0], device=x.device)
        y[..., rows, :] += anchors[..., torch.as_tensor(anchor_of[anchor_of >= 0], device=x.device), :].double()
    return y


def exact(case, seed):
    c = case
    if c["kind"] == "evict":  # rows are moved, not computed
        return None
    s = prepare(c, seed)
    if c["kind"] == "decode":
        k, v = s.k, s.v
        if s.paged:
            table = s.paged["page_table"].long()
            k, v = (x[table].reshape(s.score.shape + x.shape[-1:]) for x in (k, v))
        lens = torch.tensor(_lens(c), device="cuda")
        out, score = _exact_steps(s.q, s.kn, s.vn, k, v, s.score, lens, c["gamma"])
        return dict(out=out, score=score, k=None, v=None, pos=None, len=None)
    if c["kind"] == "embed":
        e = [_exact_rows(s.e_in[b, :s.w.in_len[b]], s.w, s.spans, b, None if s.e_text is None else s.e_text[b],
                         s.desc.capacity, s.keep) for b in range(s.w.batch)]
        return dict(e_out=torch.stack(e), pos=None, len=None)
    w, C = s.w, s.desc.capacity
    shape = (w.batch, w.layers, w.kv_heads, C, w.head_dim)
    dt = torch.float64 if c["kind"] == "fuse" else w.dtype  # a request's cache stores its rows in the cache type
    rows = []
    for x, a in ((s.k_pre, s.anchor_k), (s.v_pre, s.anchor_v)):
        y = torch.zeros(shape, dtype=dt, device="cuda")
        for b in range(w.batch):
            for l in range(w.layers):
                y[b, l] = _exact_rows(x[b, l, :, :w.in_len[b]], w, s.spans, b, None if a is None else a[b, l], C).to(dt)
        rows.append(y)
    if c["kind"] == "fuse":
        return dict(k=rows[0], v=rows[1], score=None, pos=None, len=None)
    lens = torch.tensor(_rows(w, s.spans), device="cuda")
    out, score = _exact_steps(s.q, s.kn, s.vn, rows[0], rows[1], torch.zeros(shape[:4], device="cuda"), lens, w.gamma)
    return dict(out=out, score=score, k=None, v=None, pos=None, len=None)
