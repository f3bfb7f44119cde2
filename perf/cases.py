"""What the framework is timed on: one chunk of a chunk-causal video DiT through the public entry
points, from a toy layer to a 720p layer of a 40-head model.

A case is one pass of one of these uses:

  step    the layer of a denoising call: (table,) append with or without the q/k RMS norm, attention
  append  the append alone, as when only the cache entries of a chunk are renewed
  table   the cos/sin table of a new chunk position
  stack   all layers of one chunk through ChunkStepper, eagerly
  replay  the same through ChunkStepper's CUDA graph of the chunk

The inputs have the distribution of activations behind the q/k norm, N(0, 1) per coordinate (keys
times `k_scale` for peaked attention), and the caches hold such keys and values in every slot.
"""

from __future__ import annotations

import math

import torch

import paper_2609_32518_b200 as U
from paper_2609_32518_b200.layer_loop import ChunkStepper

BF16 = torch.bfloat16
EPS = 1e-6


def _case(name, op, heads, chunk_frames, grid_h, grid_w, ring, window, starts, **more):
    case = {"name": name, "op": op, "heads": heads, "chunk_frames": chunk_frames, "grid_h": grid_h,
            "grid_w": grid_w, "ring": ring, "window": window, "starts": starts, "sink": 0,
            "sink_attend": 0, "norm": False, "table": False, "noalloc": False, "layers": 1, "k_scale": 1.0}
    case.update(more)
    return case


def listed():
    return [
        # a toy layer (2 heads, 8 x 8 tokens): what a call costs when there is next to nothing to do
        _case("tiny_step", "step", 2, 2, 8, 8, 6, 6, "4"),
        # 1.3B class (12 heads, 30 x 52 tokens), first chunk of a clip: the window is the chunk itself
        _case("first_chunk", "step", 12, 3, 30, 52, 21, 21, "0", table=True),
        # the same layer at the last chunk of a 21-frame clip, every frame attended: 32760 keys
        _case("window21", "step", 12, 3, 30, 52, 21, 21, "18", table=True),
        # 3 sink + 6 recent frames, the operating point of long clips, four layers issued eagerly
        _case("sink9_stack", "stack", 12, 3, 30, 52, 6, 6, "18", sink=3, sink_attend=3, layers=4),
        # smallest cache that holds a 9-frame window, wrapped; six layers replayed as a CUDA graph
        _case("window9_replay", "replay", 12, 3, 30, 52, 9, 9, "27", layers=6, k_scale=4.0),
        # four streams at different fill levels served together, a table per stream
        _case("streams4", "step", 12, 3, 30, 52, 21, 21, "0,6,12,18"),
        # 14B class at 720p (40 heads, 45 x 80 tokens) with the q/k norm: the largest layer
        _case("norm_14b", "step", 40, 3, 45, 80, 12, 12, "9", norm=True),
        # one of eight GPUs' share of that layer (5 heads), no allocation allowed
        _case("shard_14b", "step", 5, 3, 45, 80, 12, 12, "9", noalloc=True),
        # two streams with sizes that divide nothing: 391 tokens a frame, 5 heads, wrapped ring
        _case("ragged", "step", 5, 2, 17, 23, 7, 5, "12,8", k_scale=4.0),
        # cache entries of one chunk renewed behind the q/k norm, 1.3B class
        _case("norm_append", "append", 12, 3, 30, 52, 21, 21, "18", norm=True),
        # the same without the norm for four streams at once
        _case("append_streams4", "append", 12, 3, 30, 52, 21, 21, "0,6,12,18"),
        # table of a new chunk position at 720p
        _case("table_720p", "table", 1, 3, 45, 80, 3, 3, "120"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    """One more case of the same uses and ranges."""
    most = max(work(c)["flops"] for c in listed())
    while True:
        op = rng.choice(["step", "step", "step", "step", "append", "append", "stack", "replay", "table"])
        chunk_frames = rng.choice([1, 2, 3, 3, 4])
        grid_h, grid_w = _log_int(rng, 6, 45), _log_int(rng, 8, 80)
        heads = _log_int(rng, 1, 40)
        ring = max(chunk_frames, _log_int(rng, 3, 21))
        window = rng.choice([ring, rng.randint(chunk_frames, ring)])
        sink = rng.choice([0, 0, 0, 1, 3])
        sink_attend = rng.randint(max(0, sink - 1), sink)
        batch = rng.choice([1, 1, 1, 2, 3, 4]) if op in ("step", "append") else 1
        # chunks arrive in order from frame 0; clips reach frame 123
        starts = [chunk_frames * rng.randint(0, 120 // chunk_frames) for _ in range(batch)]
        if rng.random() < 0.25:
            starts = [chunk_frames * rng.randint(0, 21 // chunk_frames) for _ in range(batch)]
        norm = op in ("step", "append") and rng.random() < 0.5
        case = _case("", op, heads, chunk_frames, grid_h, grid_w, ring, window,
                     ",".join(str(s) for s in starts), sink=sink, sink_attend=sink_attend, norm=norm,
                     table=op == "step" and batch == 1 and rng.random() < 0.3,
                     noalloc=op == "step" and sink == 0 and rng.random() < 0.2,
                     layers=rng.randint(2, 6) if op in ("stack", "replay") else 1,
                     k_scale=rng.choice([1.0, 1.0, 1.0, 4.0]))
        del case["name"]
        tokens = grid_h * grid_w
        cache = 4 * batch * (sink + ring) * tokens * heads * 128 * case["layers"]   # bytes of K and V
        if work(case)["flops"] <= most and cache <= 1.0e9 and tokens * chunk_frames >= 128:
            return case


def _starts(case):
    return [int(s) for s in case["starts"].split(",")]


def _shape(case):
    return U.Shape.make(len(_starts(case)), case["heads"], case["chunk_frames"], case["grid_h"],
                        case["grid_w"], case["ring"])


def _normal(gen, dims, scale=1.0):
    x = torch.empty(dims, dtype=torch.float32, device="cuda").normal_(generator=gen)
    return (x * scale if scale != 1.0 else x).to(BF16)


def prepare(case, seed):
    """Activations of a chunk, the caches behind it, its table, and buffers for the results."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    shape, starts = _shape(case), _starts(case)
    batch, tokens = shape.batch, shape.chunk_tokens
    s = {"case": case, "shape": shape, "starts": starts}
    if case["op"] == "table":
        # the seed moves the chunk along the clip
        s["starts"] = [starts[0] + 1 + int(seed) % 997]
        s["cos"] = torch.empty((tokens, 64), dtype=torch.float32, device="cuda")
        s["sin"] = torch.empty_like(s["cos"])
        return s
    act = (batch, tokens, case["heads"], 128)
    cache = (batch, case["sink"] + case["ring"], shape.tokens_per_frame, case["heads"], 128)
    layers = case["layers"]
    s["qkv"] = [(_normal(gen, act), _normal(gen, act, case["k_scale"]), _normal(gen, act)) for _ in range(layers)]
    s["q_rot"] = [torch.empty(act, dtype=BF16, device="cuda") for _ in range(layers)]
    if case["op"] != "append":
        s["out"] = [torch.empty(act, dtype=BF16, device="cuda") for _ in range(layers)]
    if case["op"] in ("stack", "replay"):
        stepper = ChunkStepper(shape, layers, case["window"], case["sink"], case["sink_attend"])
        for ck, cv in zip(stepper.cache_k, stepper.cache_v):
            ck.copy_(_normal(gen, cache, case["k_scale"]))
            cv.copy_(_normal(gen, cache))
        stepper.table(starts[0])
        s["stepper"] = stepper
        if case["op"] == "replay":
            s["graph"] = stepper.chunk_graph(starts[0], s["qkv"], s["q_rot"], s["out"])
        return s
    s["cache_k"], s["cache_v"] = _normal(gen, cache, case["k_scale"]), _normal(gen, cache)
    if case["norm"]:
        wide = case["heads"] * 128
        s["gain_q"] = 1.0 + 0.2 * torch.empty(wide, device="cuda").normal_(generator=gen)
        s["gain_k"] = 1.0 + 0.2 * torch.empty(wide, device="cuda").normal_(generator=gen)
    one_table = len(set(starts)) == 1
    s["stride"] = 0 if one_table else tokens * 64
    s["cos"] = torch.empty((1 if one_table else batch, tokens, 64), dtype=torch.float32, device="cuda")
    s["sin"] = torch.empty_like(s["cos"])
    for i in range(s["cos"].shape[0]):
        U.rope_table(shape, starts[i], s["cos"][i], s["sin"][i])
    return s


def run(s):
    case, shape, starts = s["case"], s["shape"], s["starts"]
    op = case["op"]
    if op == "table":
        U.rope_table(shape, starts[0], s["cos"], s["sin"])
        return s["cos"], s["sin"]
    if op == "stack":
        s["stepper"].chunk_step(starts[0], s["qkv"], s["q_rot"], s["out"])
        return s["out"], s["q_rot"], s["stepper"].cache_k, s["stepper"].cache_v
    if op == "replay":
        s["graph"].replay()
        return s["out"], s["q_rot"], s["stepper"].cache_k, s["stepper"].cache_v
    (q, k, v), q_rot, ck, cv = s["qkv"][0], s["q_rot"][0], s["cache_k"], s["cache_v"]
    cos, sin, sink = s["cos"], s["sin"], case["sink"]
    if case["table"]:
        U.rope_table(shape, starts[0], cos, sin)
    if case["norm"]:
        U.rmsnorm_rope_kv_append(shape, sink, starts, q, k, v, s["gain_q"], s["gain_k"], EPS, cos, sin, q_rot,
                                 ck, cv, table_stream_stride=s["stride"])
    elif sink:
        U.rope_kv_append_sink(shape, sink, starts, q, k, v, cos, sin, q_rot, ck, cv,
                              table_stream_stride=s["stride"])
    else:
        U.rope_kv_append(shape, starts, q, k, v, cos, sin, q_rot, ck, cv, table_stream_stride=s["stride"])
    if op == "append":
        return q_rot, ck, cv
    out = s["out"][0]
    if sink:
        U.window_attn_sink(shape, sink, starts, case["window"], case["sink_attend"], q_rot, ck, cv, out)
    elif case["noalloc"]:
        U.window_attn_noalloc(shape, starts, case["window"], q_rot, ck, cv, out)
    else:
        U.window_attn(shape, starts, case["window"], q_rot, ck, cv, out)
    return out, q_rot, ck, cv


def work(case):
    """Bytes and operations of one pass: q, k, v and the attended cache read once, q_out, the chunk's
    cache entries and the result written once; the tables read (or written) once."""
    starts = _starts(case)
    fc, tokens = case["chunk_frames"], case["grid_h"] * case["grid_w"]
    length, wide = fc * tokens, case["heads"] * 128
    table = 2 * length * 64 * 4
    if case["op"] == "table":
        # an angle, a sine and a cosine of each distinct (position, pair), about 50 operations in double
        return {"bytes": table, "flops": 50 * (22 * fc + 21 * case["grid_h"] + 21 * case["grid_w"])}
    tables = len(set(starts)) * table
    act = len(starts) * length * wide * 2
    nbytes = 6 * act + tables + (8 * wide if case["norm"] else 0)
    flops = 3.0 * act + (4.0 * act if case["norm"] else 0.0)
    if case["op"] != "append":
        nbytes += act                                   # the result; q_out goes out and the scores need it once
        for start in starts:
            hi = start + fc
            lo = max(0, hi - case["window"])
            keys = (min(case["sink_attend"], lo) + hi - lo) * tokens
            nbytes += 4 * (keys - length) * wide        # cached K and V of the frames before the chunk
            flops += 4.0 * length * keys * wide
    return {"bytes": case["layers"] * nbytes, "flops": case["layers"] * flops}


def tolerance(case):
    if case["op"] == "append":
        return "exact"                 # float32 rotation in a fixed order, one rounding to bf16
    if case["op"] == "table":
        return {"rel": 1e-7, "max": 2.5e-7}   # double arithmetic, one rounding: a last bit may differ
    # P and the result in bf16, float32 sums: against float64 every shape is off by 2.2e-3 to 2.4e-3
    # in the 2-norm and by 8e-3 to 1.3e-2 in its worst element
    return {"rel": 1e-2, "max": 5e-2}
