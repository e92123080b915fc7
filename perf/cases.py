"""What is timed of the library: the passes that its users make, through the public binding.

A case is a dict of plain values.  Four kinds of pass:

  stream  a video stream from its start: mukv_reset, then one mukv_compress_chunk (or
          mukv_compress_chunk_scored) per chunk of frames; with ``ask`` > 0 the viewer then asks that many
          questions (mukv_retrieve, mukv_gather)
  score   mukv_score_frames_noalloc on one batch of frames
  ask     questions on a filled store: mukv_retrieve, then mukv_gather of what it selected
  ask3    the same over segments, frames and patch-level blocks: mukv_retrieve3, then mukv_gather3

Inputs are the repository's synthetic streams (scenes with a mean of their own, outlier channels), generated
on the device; the question tokens lie around the means of scenes of the stream.
"""
import math

import numpy as np
import torch

from paper_2605_22269_b200 import binding as B
from paper_2605_22269_b200.synth.cpu import StreamSpec
from paper_2605_22269_b200.synth.gpu import GpuStream

DEV = "cuda:0"

# the shape of the benchmark's streams: 28 layers, 28 query heads on 4 key heads of 128, 196 tokens per frame
FULL = dict(dtype="bf16", layers=28, q_heads=28, kv_heads=4, head_dim=128, tokens=196, keep=49, fseg=16)
# the options of a stream, at their defaults
PLAIN = dict(causal=0, low_freq=0, score_layers=1, past=0, keep_seg=0, patch=0, by_caller=0)
# how a stream ends
SILENT = dict(ask=0, k_seg=0, k_frm=0)


def listed():
    return [
        # the smallest whole session: a toy model in fp32, one chunk of eight frames, one question
        dict(name="tiny_session_fp32", kind="stream", **dict(FULL, dtype="fp32", layers=1, q_heads=2, kv_heads=2, head_dim=64,
             tokens=64, keep=16, fseg=4), **PLAIN, chunk=8, frames=8, ask=1, k_seg=1, k_frm=2),
        # a live camera: every frame is compressed as it comes, after sixteen of them somebody asks
        dict(name="live_frames", kind="stream", **FULL, **PLAIN, chunk=1, frames=16, ask=1, k_seg=1, k_frm=4),
        # the ordinary stream: chunks of sixteen frames, one minute of video
        dict(name="stream_chunks", kind="stream", **FULL, **PLAIN, chunk=16, frames=64, **SILENT),
        # another model and odd sizes: one query head per key head, 130 tokens, causal attention, chunks that cut segments
        # and a short last one
        dict(name="stream_ragged", kind="stream", **dict(FULL, layers=24, q_heads=8, kv_heads=8, head_dim=64, tokens=130, keep=33,
             fseg=5), **dict(PLAIN, causal=1), chunk=7, frames=31, **SILENT),
        # queries that also see the kept keys of the frame before the chunk
        dict(name="stream_past_keys", kind="stream", **FULL, **dict(PLAIN, past=1), chunk=16, frames=48, **SILENT),
        # scores averaged over the last five layers
        dict(name="stream_five_layers", kind="stream", **FULL, **dict(PLAIN, score_layers=5), chunk=16, frames=32, **SILENT),
        # selection over whole segments: a frame keeps as many tokens as it has among its segment's best
        dict(name="stream_segment_budget", kind="stream", **FULL, **dict(PLAIN, keep_seg=784), chunk=16, frames=64, **SILENT),
        # fp32 caches at the full size
        dict(name="stream_fp32", kind="stream", **dict(FULL, dtype="fp32"), **PLAIN, chunk=16, frames=32, **SILENT),
        # scoring inside a process that has no device memory to give
        dict(name="score_no_memory", kind="score", dtype="bf16", q_heads=28, kv_heads=4, head_dim=128, tokens=196, keep=49, frames=16,
             causal=0, low_freq=0),
        # one question on one hour of video: what the viewer waits for before the answer starts
        dict(name="ask_one", kind="ask", **FULL, frames=1800, ask=1, q_min=32, q_max=32, k_seg=4, k_frm=8, mode=B.RETR_SEMI,
             past_views=0),
        # the questions of many viewers on three hours of video: the largest
        dict(name="ask_batch", kind="ask", **FULL, frames=10800, ask=64, q_min=16, q_max=64, k_seg=8, k_frm=16, mode=B.RETR_SEMI,
             past_views=0),
        # the decode context of all three granularities for a few questions
        dict(name="ask_three_levels", kind="ask3", **FULL, patch=2, grid=14, frames=1800, ask=8, q_min=16, q_max=64, k_seg=12, k_frm=32,
             k_patch=20, mode=B.RETR_SEMI, past_views=0),
    ]


# (query heads, key heads, head size) of models of several sizes
HEADS = [(2, 2, 64), (6, 2, 64), (8, 8, 64), (14, 2, 64), (16, 2, 128), (16, 8, 64), (28, 4, 128), (28, 4, 128), (32, 8, 128)]
# square and odd token grids of a frame
TOKENS = [36, 49, 64, 77, 81, 100, 121, 130, 144, 169, 196, 196, 225, 256]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stream"] * 6 + ["score"] + ["ask"] * 3 + ["ask3"])
    hq, hkv, d = rng.choice(HEADS)
    tokens = rng.choice(TOKENS)
    keep = max(1, int(tokens * rng.choice([0.1, 0.25, 0.25, 0.25, 0.5])))
    c = dict(kind=kind, dtype="fp32" if rng.random() < 0.15 else "bf16", layers=_log_int(rng, 2, 32), q_heads=hq, kv_heads=hkv,
             head_dim=d, tokens=tokens, keep=keep, fseg=rng.randint(4, 24))
    if kind == "score":
        return dict(kind=kind, dtype=c["dtype"], q_heads=min(hq, 32), kv_heads=hkv, head_dim=d, tokens=tokens, keep=keep,
                    frames=rng.randint(1, 16), causal=int(rng.random() < 0.3), low_freq=int(rng.random() < 0.1))
    if kind == "stream":
        c.update(PLAIN, causal=int(rng.random() < 0.25), low_freq=int(rng.random() < 0.1))
        c["chunk"] = _log_int(rng, 1, 32)
        c["frames"] = min(64, c["chunk"] * rng.randint(1, 4) + rng.randint(0, c["chunk"] - 1))
        option = rng.choice(["", "", "", "past", "layers", "segments", "caller", "patch"])
        if option == "past" and keep + tokens <= 256:
            c["past"] = rng.randint(1, min(4, (256 - tokens) // keep))
        elif option == "layers":
            c["score_layers"] = min(c["layers"], rng.choice([2, 3, 5]))
        elif option == "segments":
            c["fseg"] = min(16, 4096 // tokens)
            c["chunk"] = c["fseg"] * rng.choice([1, 1, 2])
            c["frames"] = c["chunk"] * rng.randint(1, 2) + rng.randint(0, c["fseg"] - 1)
            c["keep_seg"] = keep * c["fseg"]
        elif option == "caller":
            c["by_caller"] = 1
        elif option == "patch":
            c["patch"] = rng.choice([2, 3])
        ends = rng.random() < 0.4 and option != "segments"
        c.update(dict(ask=_log_int(rng, 1, 8), k_seg=rng.randint(1, 4), k_frm=rng.randint(1, 8)) if ends else SILENT)
        return c
    c["frames"] = _log_int(rng, 64, 10800)
    c["ask"] = _log_int(rng, 1, 128)
    c["q_min"] = _log_int(rng, 1, 32)
    c["q_max"] = c["q_min"] + rng.randint(0, 40)
    c["k_seg"] = rng.randint(1, 16)
    c["k_frm"] = _log_int(rng, 1, 48)
    c["mode"] = rng.choice([B.RETR_SEMI, B.RETR_SEMI, B.RETR_PARALLEL, B.RETR_HIER])
    c["past_views"] = int(rng.random() < 0.25)
    if kind == "ask3":
        c["patch"] = rng.choice([1, 2, 3])
        c["grid"] = _grid(tokens)
        c["frames"] = min(c["frames"], 3600)
        c["k_patch"] = rng.randint(1, 32)
    # neither a larger store nor a larger context than the three-hour case has
    page = _page_bytes(c)
    c["frames"] = max(32, min(c["frames"], int(30e9 / page)))
    tokens_each = c["k_frm"] * keep + c.get("k_patch", 0) * keep // max(1, c.get("patch", 1)) ** 2 + c["k_seg"]
    c["ask"] = max(1, min(c["ask"], int(2.8e9 / (tokens_each * page / keep))))
    return c


def _grid(tokens):
    w = int(round(math.sqrt(tokens)))
    while tokens % w:
        w -= 1
    return w


def _esize(c):
    return 2 if c["dtype"] == "bf16" else 4


def _page_bytes(c):
    return 2 * c["layers"] * c["keep"] * c["kv_heads"] * c["head_dim"] * _esize(c)


# ------------------------------------------------------------------------------------------- preparation
def _spec(c, seed, frames):
    return StreamSpec(seed=1 + seed, n_layers=c.get("layers", 1), n_q_heads=c["q_heads"], n_kv_heads=c["kv_heads"],
                      head_dim=c["head_dim"], tokens_per_frame=c["tokens"], bf16=c["dtype"] == "bf16", scene_sigma=1.0,
                      frame_sigma=0.5, scene_min=10, scene_max=60, n_frames=frames)


def _config(c, chunk, **more):
    return B.make_config(n_layers=c.get("layers", 1), n_q_heads=c["q_heads"], n_kv_heads=c["kv_heads"], head_dim=c["head_dim"],
                         tokens_per_frame=c["tokens"], keep_per_frame=c["keep"], frames_per_segment=c.get("fseg", 1),
                         max_frames_per_chunk=chunk, max_frames=c["frames"], dtype=B.BF16 if c["dtype"] == "bf16" else B.FP32,
                         **more)


def _question_tokens(c, spec, seed, n, lo, hi):
    """Tokens of n questions around scene means of the last layer, and their offsets."""
    r = np.random.RandomState(seed & 0x7FFFFFFF)
    lens = r.randint(lo, hi + 1, n)
    offs = np.zeros(n + 1, dtype=np.int32)
    np.cumsum(lens, out=offs[1:])
    scenes = r.randint(0, int(spec.scene_of_frame().max()) + 1, n)
    mean = np.stack([spec.scene_mean(int(s))[-1] for s in scenes]) * np.float32(spec.scene_sigma)      # [n][Hkv][D]
    mean = torch.from_numpy(mean).to(DEV).repeat_interleave(c["q_heads"] // c["kv_heads"], dim=1)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    x = torch.randn((int(offs[-1]), c["q_heads"], c["head_dim"]), device=DEV, generator=gen)
    of = torch.from_numpy(np.repeat(np.arange(n), lens)).to(DEV)
    return (mean[of] + 0.5 * x).to(torch.bfloat16 if c["dtype"] == "bf16" else torch.float32), offs


def _answers(c, ctx, n):
    """Output buffers of mukv_retrieve and mukv_gather for n questions."""
    i32, ks, kf = torch.int32, c["k_seg"], c["k_frm"]
    stride = ctx.decode_stride_bytes(kf)
    return dict(seg=torch.full((n, ks), -1, dtype=i32, device=DEV), frm=torch.full((n, kf), -1, dtype=i32, device=DEV),
                seg_score=torch.zeros((n, ks), device=DEV), frm_score=torch.zeros((n, kf), device=DEV),
                counts=torch.zeros((n, 2), dtype=i32, device=DEV), stride=stride,
                decode=torch.zeros((n, stride // _esize(c)), dtype=ctx.torch_dtype, device=DEV),
                meta=torch.full((n, kf * c["keep"], 2), -1, dtype=i32, device=DEV))


def _prepare_stream(c, seed):
    more = dict(attn_causal=c["causal"], keep_low_freq=c["low_freq"], n_score_layers=c["score_layers"], past_frames=c["past"],
                keep_per_segment=c["keep_seg"])
    if c["patch"]:
        more.update(patch_split=c["patch"], grid_width=_grid(c["tokens"]))
    ctx = B.MukvContext(_config(c, c["chunk"], **more), DEV)
    spec = _spec(c, seed, c["frames"])
    gs = GpuStream(spec, DEV)
    T, P, layers = c["frames"], c["tokens"], c["score_layers"]
    width = P if c["keep_seg"] else c["keep"]
    kept = torch.full((T, width), -1, dtype=torch.int32, device=DEV)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    chunks, scores = [], []
    for t0 in range(0, T, c["chunk"]):
        n = min(c["chunk"], T - t0)
        q, k, v = gs.alloc(n)
        gs.fill(t0, n, q, k, v)
        if layers > 1:
            q = torch.stack([q] + [torch.randn(q.shape, device=DEV, generator=gen).to(q.dtype) for _ in range(layers - 1)])
        sc = torch.zeros((3, n, P), device=DEV)
        if c["by_caller"]:
            q, sc = torch.rand((n, P), device=DEV, generator=gen), None
        chunks.append((q, k, v, n, t0, kept[t0:t0 + n], sc))
        scores.append(sc)
    # what the stream leaves behind, as views of the store: pages, frame entries and keys, the segment entries that
    # later calls no longer change (a segment of the last chunk is pooled by the question behind it), patch-level keys
    out = [kept, ctx.region(2)[:T], ctx.region(4)[:T], ctx.region(6)[:T], ctx.region(7)[:T]]
    if c["keep_seg"]:
        full, rest = T // c["fseg"], T % c["fseg"]
        tokens = full * c["keep_seg"] + c["keep_seg"] * rest // c["fseg"]
        out += [ctx.region(0)[:tokens * 2 * c["layers"] * c["kv_heads"] * c["head_dim"]], ctx.region(10)[:T]]
    else:
        out.append(ctx.region(0)[:T])
    done = (T + c["fseg"] - 1) // c["fseg"] if c["ask"] else (chunks[-1][4] // c["fseg"])
    if done:
        out += [ctx.region(3)[:done], ctx.region(5)[:done]]
    if c["patch"]:
        out += [ctx.region(8)[:T], ctx.region(9)[:T]]
    s = dict(case=c, ctx=ctx, chunks=chunks, out=out + scores)
    if c["ask"]:
        s["qtok"], s["offs"] = _question_tokens(c, spec, seed + 1, c["ask"], 8, 32)
        s["ans"] = _answers(c, ctx, c["ask"])
    return s


def _prepare_score(c, seed):
    gs = GpuStream(_spec(c, seed, c["frames"]), DEV)
    q, k, _ = gs.alloc(c["frames"])
    gs.fill(0, c["frames"], q, k, torch.empty_like(k))
    n, P = c["frames"], c["tokens"]
    return dict(case=c, cfg=_config(c, n, attn_causal=c["causal"], keep_low_freq=c["low_freq"]), q=q, k=k[0],
                kept=torch.full((n, c["keep"]), -1, dtype=torch.int32, device=DEV), scores=torch.zeros((3, n, P), device=DEV))


def _prepare_ask(c, seed):
    T, chunk = c["frames"], 16
    more = dict(patch_split=c["patch"], grid_width=c["grid"]) if c["kind"] == "ask3" else {}
    ctx = B.MukvContext(_config(c, chunk, **more), DEV)
    spec = _spec(c, seed, T)
    gs = GpuStream(spec, DEV)
    bufs = {}
    for t0 in range(0, T, chunk):
        n = min(chunk, T - t0)
        if n not in bufs:
            bufs[n] = gs.alloc(n)
        gs.fill(t0, n, *bufs[n])
        ctx.mukv_compress_chunk(*bufs[n], n, t0)
    ctx.region(5)                                             # the last segment is pooled before anybody asks
    torch.cuda.synchronize()
    qtok, offs = _question_tokens(c, spec, seed + 1, c["ask"], c["q_min"], c["q_max"])
    n = c["ask"]
    # questions about the past of the stream see only what was stored by then
    limit = np.random.RandomState(seed & 0xFFFF).randint(max(1, T // 4), T + 1, n).astype(np.int64) if c["past_views"] else None
    s = dict(case=c, ctx=ctx, qtok=qtok, offs=offs, limit=limit)
    if c["kind"] == "ask":
        s["ans"] = _answers(c, ctx, n)
        return s
    i32, ks, kf, kp = torch.int32, c["k_seg"], c["k_frm"], c["k_patch"]
    cap = ctx.mukv_decode3_tokens(ks, kf, kp)
    stride = 2 * c["layers"] * cap * c["kv_heads"] * c["head_dim"] * _esize(c)
    s["prm"] = B.MukvRetrParams(kp, kf, ks, 0.3, 0.3, 0.0, 0, c["mode"])
    s["ans"] = dict(seg=torch.full((n, ks), -1, dtype=i32, device=DEV), frm=torch.full((n, kf), -1, dtype=i32, device=DEV),
                    pat=torch.full((n, kp), -1, dtype=i32, device=DEV), seg_score=torch.zeros((n, ks), device=DEV),
                    frm_score=torch.zeros((n, kf), device=DEV), pat_score=torch.zeros((n, kp), device=DEV),
                    counts=torch.zeros((n, 3), dtype=i32, device=DEV), stride=stride,
                    decode=torch.zeros((n, stride // _esize(c)), dtype=ctx.torch_dtype, device=DEV),
                    ntok=torch.zeros((n,), dtype=i32, device=DEV), meta=torch.full((n, cap, 2), -1, dtype=i32, device=DEV))
    return s


def prepare(case, seed):
    return dict(stream=_prepare_stream, score=_prepare_score, ask=_prepare_ask, ask3=_prepare_ask)[case["kind"]](case, seed)


# ------------------------------------------------------------------------------------------------- a pass
def _ask(s, mode, limit):
    c, ctx, a = s["case"], s["ctx"], s["ans"]
    ctx.mukv_retrieve(s["qtok"], s["offs"], limit, c["k_seg"], c["k_frm"], 0, 0.3, mode, a["seg"], a["frm"], a["seg_score"],
                      a["frm_score"], a["counts"])
    ctx.mukv_gather(a["frm"], a["counts"], c["ask"], c["k_frm"], a["decode"], a["stride"], a["meta"])
    return [a["seg"], a["frm"], a["seg_score"], a["frm_score"], a["counts"], a["decode"], a["meta"]]


def run(state):
    c = state["case"]
    if c["kind"] == "score":
        B.mukv_score_frames_noalloc(state["cfg"], state["q"], state["k"], c["frames"], state["kept"], state["scores"])
        return [state["kept"], state["scores"]]
    ctx = state["ctx"]
    if c["kind"] == "stream":
        ctx.mukv_reset()
        if c["by_caller"]:
            for x, k, v, n, t0, kept, _ in state["chunks"]:
                ctx.mukv_compress_chunk_scored(x, k, v, n, t0, kept)
        else:
            for q, k, v, n, t0, kept, sc in state["chunks"]:
                ctx.mukv_compress_chunk(q, k, v, n, t0, kept, sc)
        return state["out"] + (_ask(state, B.RETR_SEMI, None) if c["ask"] else [])
    if c["kind"] == "ask":
        return _ask(state, c["mode"], state["limit"])
    a = state["ans"]
    ctx.mukv_retrieve3(state["qtok"], state["offs"], state["limit"], state["prm"], a["seg"], a["frm"], a["pat"], a["seg_score"],
                       a["frm_score"], a["pat_score"], a["counts"])
    ctx.mukv_gather3(a["seg"], a["frm"], a["pat"], a["counts"], c["ask"], c["k_seg"], c["k_frm"], c["k_patch"], a["decode"],
                     a["stride"], a["ntok"], a["meta"])
    return [a["seg"], a["frm"], a["pat"], a["seg_score"], a["frm_score"], a["pat_score"], a["counts"], a["decode"], a["ntok"],
            a["meta"]]


# ---------------------------------------------------------------------------- what a pass cannot do without
def _score_work(c, frames, layers, past):
    """Scoring: the queries and keys of the scoring layers read, the two products of Eq. 1 counted once, a fast
    Fourier transform per key vector."""
    P, d = c["tokens"], c["head_dim"]
    read = layers * frames * P * (c["q_heads"] + c["kv_heads"]) * d * _esize(c)
    flops = layers * frames * (2.0 * c["q_heads"] * P * (P + past) * d + 2.5 * c["kv_heads"] * P * d * math.log2(d))
    return read, flops


def _ask_work(c, ask, tokens_q, tokens_ctx, frames, patches):
    """Questions: their tokens and the keys of every visible block read, the selected context read and written."""
    C = c["kv_heads"] * c["head_dim"]
    rows = frames + (frames + c["fseg"] - 1) // c["fseg"] + patches
    moved = 2 * ask * tokens_ctx * (_page_bytes(c) // c["keep"])
    return tokens_q * c["q_heads"] * c["head_dim"] * _esize(c) + rows * C * 4 + moved, 2.0 * ask * rows * C


def work(case):
    c = case
    if c["kind"] == "score":
        read, flops = _score_work(c, c["frames"], 1, 0)
        return {"bytes": read + c["frames"] * (4 * c["keep"] + 12 * c["tokens"]), "flops": flops}
    C = c["kv_heads"] * c["head_dim"]
    if c["kind"] == "stream":
        T = c["frames"]
        kept = T * _page_bytes(c)
        entries = 2 * c["layers"] * C * 4 * (T + (T + c["fseg"] - 1) // c["fseg"])
        if c["by_caller"]:
            read, flops = T * c["tokens"] * 4, 0.0
            seen = 0
        else:
            read, flops = _score_work(c, T, c["score_layers"], c["past"] * c["keep"])
            read += T * c["tokens"] * 12                                   # the scores are written
            seen = c["score_layers"] * kept // (2 * c["layers"])           # kept keys that scoring has read already
        b = read + 2 * kept - seen + entries + T * (8 * c["keep"] + 12 * C)
        if c["patch"]:
            b += T * c["patch"] ** 2 * C * 4
        if c["ask"]:
            qb, qf = _ask_work(c, c["ask"], c["ask"] * 20, min(c["k_frm"], T) * c["keep"], T, 0)
            b, flops = b + qb, flops + qf
        return {"bytes": b, "flops": flops}
    patches, tokens_ctx = 0, min(c["k_frm"], c["frames"]) * c["keep"]
    if c["kind"] == "ask3":
        patches = c["frames"] * c["patch"] ** 2
        tokens_ctx += c["k_seg"] + c["k_patch"] * c["keep"] // c["patch"] ** 2
    b, f = _ask_work(c, c["ask"], c["ask"] * (c["q_min"] + c["q_max"]) / 2, tokens_ctx, c["frames"], patches)
    return {"bytes": b, "flops": f}


def tolerance(case):
    # Ids, counts and copied rows do not depend on rounding: a choice that single precision cannot make safely is made in
    # double precision.  Scores and entries are 32-bit sums of up to a few thousand terms.
    if case["kind"] == "ask3":
        return {"rel": 1e-5, "max": 0.01}                     # a summary token may round to the next bf16 value
    return {"rel": 1e-5}
