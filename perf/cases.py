"""The work that programs give this library, as cases that can be timed and compared.

A case is one pass through the public entry points of `paper_2411_10803_b200.binding`:

  filter   one pruning layer in one call (scores, selection, compaction)
  staged   the same step as its three calls, as a program makes them that wants the kept indices in between
  layers   a chain of pruning layers on a ragged batch, each on what the layer before it kept
  cache    the decode-stage rebuild of the K / V caches of all later layers
  vision   the vision-encoding stage: spatial merge of the encoder's tokens, key set from its [CLS] attention

Sizes are those of `synth.WORKLOADS` (336 x 336 images of 576 tokens, high-resolution inputs of 2880,
8 video frames of 2048, 7B and 13B head counts) and of the side measurements of `bench.py`, plus generic
ones that no tile divides.
"""
import math

import torch

from paper_2411_10803_b200 import binding as md

HEAD_DIM = 128
BF16 = 2
MOST_BYTES = 750e6      # what a drawn case may move


def _filter(name, op="filter", **kw):
    case = {"op": op, "batch": 1, "n_vis": 576, "n_txt": 64, "n_heads": 32, "vis_start": 0, "keep": 64, "key_cnt": 32,
            "frames": 1, "threshold": False, "per_head_max": False, "causal": True, "token_major": False}
    case.update(kw)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # one image and one question: the smallest call, all latency
        _filter("one_image", n_txt=32, key_cnt=16),
        # a server's ordinary batch of images at the mildest budget
        _filter("batch16_keep192", batch=16, keep=192),
        # the throughput point of the benchmark: a full batch, the tightest budget
        _filter("batch64_keep64", batch=64),
        # high-resolution images: few requests, long sequences
        _filter("highres_2880", batch=8, n_vis=2880, keep=320, key_cnt=64),
        # video: keys that repeat from frame to frame, long questions
        _filter("video_2048", batch=8, n_vis=2048, n_txt=96, keep=256, key_cnt=64, frames=8),
        # the larger model's head count at a full batch, the longest questions: the largest filter call
        _filter("heads40_batch64", batch=64, n_txt=128, n_heads=40),
        # nothing divides: system prompt in front, odd counts, K / V as the projection wrote them
        # (token-major), and the rule exactly as printed (thresholds instead of a budget)
        _filter("odd_threshold", batch=5, n_vis=1451, n_txt=43, vis_start=35, key_cnt=21, threshold=True, token_major=True),
        # the other reading of the per-token maximum over heads, medium batch
        _filter("per_head_max", batch=24, keep=128, per_head_max=True),
        # three calls instead of one, at a batch that does not fill the GPU evenly
        _filter("staged_batch12", op="staged", batch=12, keep=144),
        # images that the spatial merge has left with 60 to 95 % of their tokens, through three pruning layers
        {"name": "layers_ragged", "op": "layers", "batch": 32, "n_vis": 576, "n_txt": 64, "n_heads": 32, "vis_start": 0,
         "keep": 192, "keep2": 128, "keep3": 64, "key_cnt": 32},
        # the caches of the thirty later layers once the last pruning layer has spoken
        {"name": "cache_30_layers", "op": "cache", "n_layers": 30, "batch": 8, "n_heads": 32, "held": 64, "vis_start": 0,
         "n_tail": 64},
        # the vision encoder's side of a batch of 336 x 336 images
        {"name": "vision_batch64", "op": "vision", "batch": 64, "grid": 24, "channels": 1024, "n_heads": 16, "head_dim": 64,
         "key_max": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choices(["filter", "staged", "layers", "cache", "vision"], [60, 8, 12, 8, 12])[0]
    heads = rng.choice([8, 16, 24, 28, 32, 32, 40])
    if op in ("filter", "staged"):
        n_vis = _log(rng, 64, 4096)
        case = _filter(None, op=op, batch=_log(rng, 1, 64), n_vis=n_vis, n_txt=rng.randint(8, 128), n_heads=heads,
                       vis_start=rng.choice([0, 0, 35, rng.randint(1, 64)]), keep=max(4, int(n_vis * rng.uniform(0.05, 0.4))),
                       threshold=rng.random() < 0.15, per_head_max=op == "filter" and rng.random() < 0.1,
                       causal=rng.random() < 0.9, token_major=rng.random() < 0.2)
        case["key_cnt"] = rng.randint(0, case["keep"] // 2)
    elif op == "layers":
        n_vis = _log(rng, 144, 1024)
        keep = max(12, int(n_vis * rng.uniform(0.2, 0.4)))
        case = {"op": op, "batch": _log(rng, 1, 32), "n_vis": n_vis, "n_txt": rng.randint(8, 96), "n_heads": heads,
                "vis_start": rng.choice([0, 35]), "keep": keep, "keep2": 2 * keep // 3, "keep3": keep // 3,
                "key_cnt": rng.randint(0, keep // 4)}
    elif op == "cache":
        case = {"op": op, "n_layers": rng.randint(8, 38), "batch": _log(rng, 1, 32), "n_heads": heads,
                "held": _log(rng, 32, 320), "vis_start": rng.choice([0, 35]), "n_tail": rng.randint(8, 128)}
    else:
        case = {"op": op, "batch": _log(rng, 1, 96), "grid": 2 * rng.randint(6, 24), "channels": 8 * rng.randint(64, 176),
                "n_heads": rng.choice([12, 16]), "head_dim": rng.choice([64, 72, 80, 88]), "key_max": rng.choice([32, 64, 128])}
    while case["batch"] > 1 and work(case)["bytes"] > MOST_BYTES:
        case["batch"] = max(1, case["batch"] * 3 // 4)
    while op == "cache" and work(case)["bytes"] > MOST_BYTES:
        case["n_layers"] = max(1, case["n_layers"] * 3 // 4)
    return case


# ---- inputs ---------------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)


def _some_of(g, batch, n, count):
    """`count` distinct indices below n per request, ascending, int32 [batch, max(count, 1)] and the counts."""
    idx = torch.full((batch, max(count, 1)), -1, dtype=torch.int32, device="cuda")
    if count:
        order = torch.rand((batch, n), generator=g, device="cuda").argsort(dim=1)
        idx[:, :count] = order[:, :count].sort(dim=1).values.to(torch.int32)
    return idx, torch.full((batch,), count, dtype=torch.int32, device="cuda")


def _attention(g, batch, heads, n_txt, length, vis_start, n_vis, frames=1, token_major=False):
    """Queries and keys whose attention is spread the way trained models spread it: every token has a
    salience that all heads and questions share (the log of its attention varies with deviation 1 from
    token to token), on top of which each head and query sees its own noise."""
    direction = torch.nn.functional.normalize(torch.randn((batch, heads, 1, HEAD_DIM), generator=g, device="cuda"), dim=-1)
    q = (_normal(g, batch, heads, n_txt, HEAD_DIM) + 4.0 * direction).to(torch.bfloat16)
    noise = _normal(g, batch, heads, length, HEAD_DIM)
    salience = torch.randn((batch, 1, length, 1), generator=g, device="cuda")
    if frames > 1:      # what a patch shows changes slowly from frame to frame
        per = n_vis // frames
        for t in (noise, salience):
            v = t[:, :, vis_start:vis_start + frames * per].unflatten(2, (frames, per))
            for f in range(1, frames):
                v[:, :, f] = 0.9 * v[:, :, f - 1] + math.sqrt(1.0 - 0.81) * v[:, :, f]
    k = torch.empty((batch, length, heads, HEAD_DIM), dtype=torch.bfloat16, device="cuda").transpose(1, 2) if token_major \
        else torch.empty((batch, heads, length, HEAD_DIM), dtype=torch.bfloat16, device="cuda")
    k.copy_(noise + (math.sqrt(HEAD_DIM) / 4.0) * (salience * direction).to(torch.bfloat16))
    return q, k


def _prepare_filter(c, g):
    B, H, M, N, vs = c["batch"], c["n_heads"], c["n_vis"], c["n_txt"], c["vis_start"]
    L = vs + M + N
    q, k = _attention(g, B, H, N, L, vs, M, c["frames"], c["token_major"])
    v = _normal(g, B, L, H, HEAD_DIM).transpose(1, 2) if c["token_major"] else _normal(g, B, H, L, HEAD_DIM)
    hidden = _normal(g, B, L, H * HEAD_DIM)
    key_idx, key_cnt = _some_of(g, B, M, c["key_cnt"])
    strides = {}
    if c["token_major"]:
        for t in ("k", "v"):
            strides.update({t + "_stride_b": L * H * HEAD_DIM, t + "_stride_h": HEAD_DIM, t + "_stride_l": H * HEAD_DIM})
    f = md.Filter(md.Config(
        batch=B, n_heads=H, hidden=H * HEAD_DIM, seq_len=L, vis_start=vs, n_vis=M, txt_start=vs + M, n_txt=N,
        causal=int(c["causal"]), mode=md.MUSTDROP_MODE_THRESHOLD if c["threshold"] else md.MUSTDROP_MODE_BUDGET,
        budget=0 if c["threshold"] else c["keep"], key_max=c["key_cnt"],
        flags=md.MUSTDROP_FLAG_PER_HEAD_MAX if c["per_head_max"] else 0, **strides))
    keys = (key_idx, key_cnt) if c["key_cnt"] else (None, None)
    return {"op": c["op"], "filter": f, "inputs": (q, k, v, hidden) + keys}


def _prepare_layers(c, g):
    B, H, N, vs = c["batch"], c["n_heads"], c["n_txt"], c["vis_start"]
    low = max(int(0.6 * c["n_vis"]), 1)
    vis_cnt = torch.randint(low, int(0.95 * c["n_vis"]) + 1, (B,), generator=g, device="cuda").to(torch.int32)
    key_idx, key_cnt = _some_of(g, B, low, c["key_cnt"])
    state = {"op": "layers", "vis_cnt": vis_cnt, "keys": (key_idx, key_cnt) if c["key_cnt"] else (None, None), "layers": []}
    capacity = c["n_vis"]
    for keep in (c["keep"], c["keep2"], c["keep3"]):
        L = vs + capacity + N
        q, k = _attention(g, B, H, N, L, vs, capacity)
        f = md.Filter(md.Config(batch=B, n_heads=H, hidden=H * HEAD_DIM, seq_len=L, vis_start=vs, n_vis=capacity,
                                txt_start=vs + capacity, n_txt=N, budget=keep, key_max=c["key_cnt"],
                                flags=md.MUSTDROP_FLAG_REBUILD_SEQUENCE))
        state["layers"].append((f, q, k, _normal(g, B, H, L, HEAD_DIM), _normal(g, B, L, H * HEAD_DIM)))
        capacity = keep
    return state


def _prepare_cache(c, g):
    n, B, H, held, vs, tail = c["n_layers"], c["batch"], c["n_heads"], c["held"], c["vis_start"], c["n_tail"]
    rows = vs + held + tail
    ids, _ = _some_of(g, B, 9 * held, held)
    # of the tokens a layer holds, 60 to 80 % are still wanted after the last pruning layer
    few_cnt = torch.randint(int(0.6 * held), int(0.8 * held) + 1, (B,), generator=g, device="cuda")
    order = torch.rand((B, held), generator=g, device="cuda").argsort(dim=1)
    wanted = torch.zeros((B, held), dtype=torch.bool, device="cuda")
    wanted.scatter_(1, order, torch.arange(held, device="cuda").expand(B, held) < few_cnt[:, None])
    few = torch.where(wanted, ids, torch.full_like(ids, 1 << 30)).sort(dim=1).values
    few = torch.where(few == 1 << 30, torch.full_like(few, -1), few).contiguous()
    out = [torch.zeros((n, B, H, rows, HEAD_DIM), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
    return {"op": "cache", "caches": [_normal(g, n, B, H, rows, HEAD_DIM) for _ in range(2)], "out": out,
            "ids": ids.expand(n, B, held).contiguous(), "cnt": torch.full((n, B), held, dtype=torch.int32, device="cuda"),
            "few": few, "few_cnt": few_cnt.to(torch.int32), "workspace": torch.zeros(256, dtype=torch.uint8, device="cuda"),
            "sizes": dict(n_layers=n, batch=B, n_heads=H, rows_in=rows, vis_start=vs, n_tail=tail, ids_max=held, cap=held)}


def _prepare_vision(c, g):
    B, grid, C, H, D = c["batch"], c["grid"], c["channels"], c["n_heads"], c["head_dim"]
    M, half = grid * grid, grid // 2
    tokens = _normal(g, B, half, 2, half, 2, C)
    # 30 % of the 2 x 2 windows show nothing new: one vector, four times, and a little noise
    flat = torch.rand((B, half, 1, half, 1, 1), generator=g, device="cuda") < 0.3
    tokens = torch.where(flat, _normal(g, B, half, 1, half, 1, C) + 0.05 * tokens, tokens).view(B, M, C)
    q = _normal(g, B, H, D)
    k = _normal(g, B, H, M, D)
    # a twentieth of the keys stand out to every head
    outlier, _ = _some_of(g, B, M, max(1, M // 20))
    pull = 0.6 * math.sqrt(D) * torch.nn.functional.normalize(q.float(), dim=-1)
    mark = torch.zeros((B, M), device="cuda").scatter_(1, outlier.long(), 1.0)
    k = (k + (mark[:, None, :, None] * pull[:, :, None, :]).to(torch.bfloat16)).contiguous()
    i32, f32 = dict(dtype=torch.int32, device="cuda"), dict(dtype=torch.float32, device="cuda")
    return {"op": "vision", "sizes": (B, grid, 2, C, 0.8), "heads": (B, H, D, M, c["key_max"]), "tokens": tokens, "q": q, "k": k,
            "merged": torch.zeros((B, M, C), dtype=torch.bfloat16, device="cuda"), "slots": torch.full((B, M), -1, **i32),
            "merged_cnt": torch.zeros((B,), **i32), "sim": torch.zeros((B, half * half), **f32),
            "a_cls": torch.zeros((B, M), **f32), "mu": torch.zeros((B,), **f32),
            "key_idx": torch.full((B, c["key_max"]), -1, **i32), "key_cnt": torch.zeros((B,), **i32)}


def prepare(case, seed):
    make = {"filter": _prepare_filter, "staged": _prepare_filter, "layers": _prepare_layers, "cache": _prepare_cache,
            "vision": _prepare_vision}
    return make[case["op"]](case, _generator(seed))


# ---- one pass ---------------------------------------------------------------------------------------
def _must(status):
    if status != md.MUSTDROP_OK:
        raise RuntimeError(md.mustdrop_status_string(status))


def _outputs(f):
    return {"g": f.g, "i": f.i, "kept_idx": f.kept_idx, "kept_cnt": f.kept_cnt, "hidden": f.hidden_out, "k": f.k_out,
            "v": f.v_out}


def run(s):
    if s["op"] == "filter":
        s["filter"].filter(*s["inputs"])
        return _outputs(s["filter"])
    if s["op"] == "staged":
        q, k, v, hidden, key_idx, key_cnt = s["inputs"]
        f = s["filter"]
        f.score(q, k)
        f.select(key_idx, key_cnt, want_s=False)
        f.compact(hidden, k, v)
        return _outputs(f)
    if s["op"] == "layers":
        (key_idx, key_cnt), cnt, orig = s["keys"], s["vis_cnt"], None
        for f, q, k, v, hidden in s["layers"]:
            f.filter_layer(q, k, v, hidden, key_idx, key_cnt, vis_cnt=cnt, orig_idx=orig)
            if key_idx is not None:
                key_idx, key_cnt = f.key_idx_out, f.key_cnt_out
            cnt, orig = f.kept_cnt, f.orig_out
        return [dict(_outputs(f), orig=f.orig_out) for f, *_ in s["layers"]]
    if s["op"] == "cache":
        _must(md.mustdrop_cache_compact(*s["caches"], s["ids"], s["cnt"], s["few"], s["few_cnt"], *s["out"], s["workspace"],
                                        **s["sizes"]))
        return s["out"]
    _must(md.mustdrop_spatial_merge(*s["sizes"], s["tokens"], s["merged"], s["slots"], s["merged_cnt"], s["sim"]))
    _must(md.mustdrop_key_set(*s["heads"], s["q"], s["k"], s["a_cls"], s["mu"], s["key_idx"], s["key_cnt"]))
    return [s[n] for n in ("merged", "slots", "merged_cnt", "sim", "a_cls", "mu", "key_idx", "key_cnt")]


# ---- what a pass cannot do without ------------------------------------------------------------------
def _layer_work(batch, heads, length, n_txt, n_vis, rows_read, rows_written):
    """Keys, queries, the kept rows of hidden and V read (those of K have been read already), the
    kept rows of all three written, the scores written; the logits' multiply-adds."""
    row = heads * HEAD_DIM * BF16
    return {"bytes": batch * (row * (length + n_txt) + 2 * rows_read * row + 3 * rows_written * row + 8 * n_vis),
            "flops": batch * 2.0 * heads * n_txt * length * HEAD_DIM}


def work(case):
    c = case
    B, H = c["batch"], c["n_heads"]
    if c["op"] in ("filter", "staged"):
        # (as printed, the rule keeps about a third of the tokens at these inputs)
        kept = 0.33 * c["n_vis"] if c["threshold"] else c["keep"]
        return _layer_work(B, H, c["vis_start"] + c["n_vis"] + c["n_txt"], c["n_txt"], c["n_vis"], kept, kept)
    if c["op"] == "layers":
        total, tokens = {"bytes": 0.0, "flops": 0.0}, 0.775 * c["n_vis"]
        for keep, capacity in ((c["keep"], c["n_vis"]), (c["keep2"], c["keep"]), (c["keep3"], c["keep2"])):
            rows = c["vis_start"] + min(keep, tokens) + c["n_txt"]
            w = _layer_work(B, H, c["vis_start"] + tokens + c["n_txt"], c["n_txt"], capacity, rows, rows)
            total = {n: total[n] + w[n] for n in total}
            tokens = min(keep, tokens)
        return total
    if c["op"] == "cache":
        rows = c["vis_start"] + 0.7 * c["held"] + c["n_tail"]
        return {"bytes": 2.0 * 2 * c["n_layers"] * B * H * rows * HEAD_DIM * BF16, "flops": 0.0}
    M, C, D = c["grid"] ** 2, c["channels"], c["head_dim"]
    # 30 % of the windows leave one row of four
    return {"bytes": B * (M * C * BF16 * (1 + 0.775) + H * (M + 1) * D * BF16 + M * (4 + 4 + 1)),
            "flops": B * (5.0 * M * C + 2.0 * H * M * D)}


def tolerance(case):
    if case["op"] == "cache":
        return "exact"
    # Rows are copied, so only scores can differ: means of thousands of 32-bit terms.  Against the
    # two-pass kernel, which sums in another order, they are off by up to 2.1e-7 (4.4e-5 where the
    # per-head maxima are kept in 11 bits); the vision stage's by up to 4.3e-7 against 64 bits.
    if case["op"] == "vision":
        return {"rel": 2e-6}
    return {"rel": 2e-4 if case.get("per_head_max") else 1e-6}
