"""Cases of the VideoMLA attention layer for measuring: sizes, inputs, one pass, work and exact values.

A case names one call (or the calls of one layer) that a program with a
latent cache makes for every chunk of a rollout, at one size:

  append     mla_cache_append: the chunk's tokens into the cache
  query      mla_query_prologue: the chunk's absorbed queries
  attention  mla_attention_forward: the chunk against the valid window
  window     mla_attention_window_forward: the same over a sink + FIFO window
  output     mla_output_projection: the latent output back to the model width
  dense      mla_decompress_window, then mla_dense_attention_forward on it
  layer      append, query, attention and output, as a backbone calls them

Sizes: latent grids of 8 x 8 to 30 x 52 tokens per frame, chunks of 1 to 3
frames, windows of 4 to 21 frames (partly filled at the start of a rollout,
wrapped later), batches of 1 to 16, d_c in {64, 128, 192, 256, 512} and
d_r in {32, 64}; hidden 1536, 12 heads of 128, d_q 768. Inputs follow the
repository's synthetic recipe: unit-normal activations and latents, weights
of variance 1 / fan-in, all bf16.
"""

import math

import torch

from paper_2605_30351_gb300 import synth
from paper_2605_30351_gb300 import videomla as V

HIDDEN, HEADS, HEAD_DIM, D_Q = 1536, 12, 128, 768
EPS = 1e-6
ROPE = {32: ((6, 5, 5), (44, 42, 42)), 64: ((12, 10, 10), (64, 64, 64))}
ROPE_LEN = 1024


def _case(name, op, *, batch=1, grid=(30, 52), frames=3, window=21, sink=0, at=21, d_c=192, d_r=32):
    """at: frames written once the chunk is in the cache (the rollout's position)."""
    case = {"op": op, "batch": batch, "grid_h": grid[0], "grid_w": grid[1], "frames": frames,
            "window": window, "sink": sink, "at": at, "d_c": d_c, "d_r": d_r}
    return {"name": name, **case} if name else case


def listed():
    return [
        # one 64-token frame into a four-frame cache: a small model or a unit
        # test of a larger program, all latency
        _case("append_small", "append", grid=(8, 8), frames=1, window=4, at=4),
        # every denoising step of every block at batch 1 rewrites its chunk
        _case("append_chunk", "append"),
        # a server with 16 sequences in flight, their rings wrapped
        _case("append_batch", "append", batch=16, at=300),
        # one small frame against its small window: all latency
        _case("attention_small", "attention", grid=(8, 8), frames=1, window=4, at=4),
        # previews at half the resolution (15 x 26 latents), ragged row and key tiles
        _case("attention_lowres", "attention", grid=(15, 26)),
        # the paper's layer: 4,680 query tokens x 12 heads against 32,760 keys
        _case("attention_chunk", "attention"),
        # the smallest latent of the d_c ablation
        _case("attention_dc64", "attention", d_c=64),
        # the largest latent of the ablation, with the wide positional key
        _case("attention_dc512", "attention", d_c=512, d_r=64),
        # long rollout: 1 sink + 6 newest frames, batch 4, keys rotated at use
        _case("window_rollout", "window", batch=4, window=7, sink=1, at=960),
        # queries of four sequences' chunks
        _case("query_rollout", "query", batch=4, at=960),
        # the non-absorbed way: expand the window to per-head K and V, attend densely
        _case("dense_chunk", "dense"),
        # the whole attention layer of one denoising step
        _case("layer_chunk", "layer"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo - 0.49), math.log(hi + 0.49)))))))


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        op = rng.choice(["append", "append", "query", "attention", "attention", "attention",
                         "window", "output", "dense", "layer"])
        sink = rng.choice([1, 1, 2]) if op == "window" else 0
        window = _log_int(rng, 4 + sink, 9 if sink else 21)
        frames = rng.randint(1, 3)
        at = rng.randint(frames, window) if rng.random() < 0.4 else rng.randint(window, 960)
        case = _case(None, op, batch=_log_int(rng, 1, 16 if op == "append" else 4),
                     grid=(_log_int(rng, 8, 30), _log_int(rng, 8, 52)), frames=frames,
                     window=window, sink=sink, at=at,
                     d_c=rng.choice([64, 128, 192, 192, 256] + ([] if op == "dense" else [512])),
                     d_r=rng.choice([32, 32, 64]))
        if work(case)["flops"] <= most:
            return case


# ------------------------------------------------------------------- shapes
def _sizes(case):
    T = case["grid_h"] * case["grid_w"]
    held = min(case["at"], case["window"])
    return {"T": T, "tok": T * case["frames"], "slots": T * case["window"], "keys": T * held}


def _slot_frames(case):
    """Frame held in each frame slot (-1: none), the sinks first, then FIFO."""
    W, S, fw = case["window"], case["sink"], case["at"]
    out = [-1] * W
    for f in range(fw):
        out[f if f < S else S + (f - S) % (W - S)] = f
    return out


def _config(case, flags=0):
    pairs, dims = ROPE[case["d_r"]]
    w = synth.Workload("case", hidden=HIDDEN, heads=HEADS, head_dim=HEAD_DIM, d_c=case["d_c"],
                       d_r=case["d_r"], d_q=D_Q, rope_pairs=pairs, rope_axis_dims=dims,
                       rope_table_len=ROPE_LEN, grid_h=case["grid_h"], grid_w=case["grid_w"],
                       window_frames=case["window"], chunk_frames=case["frames"],
                       batch=case["batch"], last_frame=case["at"], rms_eps=EPS,
                       sink_frames=case["sink"])
    return V.make_config(w, flags)


# ------------------------------------------------------------------- inputs
def _inputs(case, seed):
    """The tensors a program has before the call, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    z = _sizes(case)
    B, H, dc, dr, tok = case["batch"], HEADS, case["d_c"], case["d_r"], z["tok"]
    op = case["op"]

    def normal(*shape, std=1.0):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).mul_(std).bfloat16()

    t = {}
    # (t, h, w) of the chunk's tokens: absolute frame, raster position
    f = torch.arange(case["at"] - case["frames"], case["at"], device="cuda", dtype=torch.int32)
    hw = torch.stack(torch.meshgrid(
        torch.arange(case["grid_h"], device="cuda", dtype=torch.int32),
        torch.arange(case["grid_w"], device="cuda", dtype=torch.int32), indexing="ij"), -1).view(-1, 2)
    pos = torch.cat([f.repeat_interleave(z["T"])[:, None], hw.repeat(case["frames"], 1)], 1)
    t["pos"] = pos.expand(B, -1, -1).contiguous()
    t["hw"] = hw.contiguous()
    if op in ("append", "query", "layer"):
        t["x"] = normal(B, tok, HIDDEN)
    if op in ("append", "layer"):
        t["w_dkv"] = normal(dc, HIDDEN, std=HIDDEN ** -0.5)
        t["w_kr"] = normal(dr, HIDDEN, std=HIDDEN ** -0.5)
        t["gamma"] = (1 + normal(dc, std=0.1)).bfloat16()
    if op in ("query", "layer"):
        t["w_dq"] = normal(D_Q, HIDDEN, std=HIDDEN ** -0.5)
        dn = HEAD_DIM - dr
        t["w_qcat"] = torch.cat([normal(H * dc, D_Q, std=(dn / (D_Q * dc)) ** 0.5),
                                 normal(H * dr, D_Q, std=D_Q ** -0.5)])
    if op in ("output", "layer"):
        t["w_b"] = normal(HIDDEN, H * dc, std=(H * dc) ** -0.5)
    if op == "output":
        t["o_lat"] = normal(B, tok, H, dc, std=0.2)
    if op != "query" and op != "output":
        t["c"] = normal(B, z["slots"], dc)
        t["kr"] = normal(B, z["slots"], dr)
    if op in ("attention", "window"):
        t["q_c"] = normal(B, tok, H, dc, std=((HEAD_DIM - dr) / dc) ** 0.5)
        t["q_r"] = normal(B, tok, H, dr)
    if op == "dense":
        t["q"] = normal(B, tok, H, HEAD_DIM)
        t["w_uk"] = normal(H, HEAD_DIM - dr, dc, std=dc ** -0.5)
        t["w_uv"] = normal(H, HEAD_DIM, dc, std=dc ** -0.5)
    return t


def prepare(case, seed):
    t = _inputs(case, seed)
    z = _sizes(case)
    cfg = _config(case)
    B, dc, dr, tok = case["batch"], case["d_c"], case["d_r"], z["tok"]
    s = {"case": case, "cfg": cfg, "t": t}

    def empty(*shape):
        return torch.empty(shape, dtype=torch.bfloat16, device="cuda")

    if "c" in t:
        s["cache"] = V.LatentCache(cfg)
        s["cache"].c.copy_(t.pop("c"))
        s["cache"].kr.copy_(t.pop("kr"))
        s["cache"].frames_written = case["at"]
    if case["op"] in ("attention", "window", "layer"):
        s["o_lat"] = empty(B, tok, HEADS, dc)
    if case["op"] in ("query", "layer"):
        s["q_c"], s["q_r"] = empty(B, tok, HEADS, dc), empty(B, tok, HEADS, dr)
        s["ws"] = torch.empty(V.mla_query_workspace_bytes(cfg, tok), dtype=torch.uint8, device="cuda")
    if case["op"] == "window":
        s["ws"] = torch.empty(V.mla_window_workspace_bytes(cfg, tok), dtype=torch.uint8, device="cuda")
    if case["op"] in ("output", "layer"):
        s["y"] = empty(B, tok, HIDDEN)
    if case["op"] == "dense":
        s["k"] = empty(B, HEADS, z["slots"], HEAD_DIM)
        s["v"] = empty(B, HEADS, z["slots"], HEAD_DIM)
        s["o"] = empty(B, tok, HEADS, HEAD_DIM)
    return s


# ----------------------------------------------------------------- one pass
def run(s):
    case, cfg, t = s["case"], s["cfg"], s["t"]
    op = case["op"]
    if op == "append":
        cache = s["cache"]
        V.mla_cache_append(cache, t["x"], t["w_dkv"], t["gamma"], t["w_kr"], t["pos"],
                           case["at"] - case["frames"], case["frames"])
        return {"c": cache.c, "kr": cache.kr}
    if op == "query":
        V.mla_query_prologue(cfg, t["x"], t["w_dq"], t["w_qcat"], s["ws"], s["q_c"], s["q_r"])
        return {"q_c": s["q_c"], "q_r": s["q_r"]}
    if op == "attention":
        V.mla_attention_forward(s["cache"], t["q_c"], t["q_r"], t["pos"], s["o_lat"])
        return {"o": s["o_lat"]}
    if op == "window":
        V.mla_attention_window_forward(s["cache"], t["q_c"], t["q_r"], t["pos"], t["hw"], s["ws"],
                                       s["o_lat"])
        return {"o": s["o_lat"]}
    if op == "output":
        V.mla_output_projection(cfg, t["o_lat"], t["w_b"], s["y"])
        return {"y": s["y"]}
    if op == "dense":
        V.mla_decompress_window(s["cache"], t["w_uk"], t["w_uv"], s["k"], s["v"])
        V.mla_dense_attention_forward(cfg, t["q"], s["k"], s["v"], _sizes(case)["keys"], s["o"])
        return {"k": s["k"], "v": s["v"], "o": s["o"]}
    cache = s["cache"]  # layer
    V.mla_cache_append(cache, t["x"], t["w_dkv"], t["gamma"], t["w_kr"], t["pos"],
                       case["at"] - case["frames"], case["frames"])
    V.mla_query_prologue(cfg, t["x"], t["w_dq"], t["w_qcat"], s["ws"], s["q_c"], s["q_r"])
    V.mla_attention_forward(cache, s["q_c"], s["q_r"], t["pos"], s["o_lat"])
    V.mla_output_projection(cfg, s["o_lat"], t["w_b"], s["y"])
    return {"c": cache.c, "kr": cache.kr, "y": s["y"]}


# --------------------------------------------------------------------- work
def work(case):
    """Each input read once, each output written once; 2 flops per multiply-add."""
    z = _sizes(case)
    B, H, dc, dr, tok, keys = case["batch"], HEADS, case["d_c"], case["d_r"], z["tok"], z["keys"]
    M = B * tok
    n_qcat = H * (dc + dr)
    x = M * HIDDEN * 2
    if case["op"] == "append":
        return {"bytes": x + (dc + dr) * HIDDEN * 2 + M * ((dc + dr) * 2 + 12),
                "flops": 2 * M * HIDDEN * (dc + dr)}
    if case["op"] == "query":
        return {"bytes": x + D_Q * HIDDEN * 2 + n_qcat * D_Q * 2 + M * n_qcat * 2,
                "flops": 2 * M * D_Q * (HIDDEN + n_qcat)}
    if case["op"] in ("attention", "window"):
        return {"bytes": B * keys * (dc + dr) * 2 + M * H * (2 * dc + dr) * 2 + M * 12,
                "flops": B * tok * H * keys * (4 * dc + 2 * dr)}
    if case["op"] == "output":
        return {"bytes": M * H * dc * 2 + HIDDEN * H * dc * 2 + x,
                "flops": 2 * M * HIDDEN * H * dc}
    if case["op"] == "dense":
        kv = B * z["slots"]
        up = H * (2 * HEAD_DIM - dr)
        return {"bytes": kv * (dc + dr) * 2 + up * dc * 2 + 2 * kv * H * HEAD_DIM * 2 +
                         2 * B * keys * H * HEAD_DIM * 2 + 2 * M * H * HEAD_DIM * 2,
                "flops": 2 * kv * up * dc + B * tok * H * keys * 4 * HEAD_DIM}
    # layer: x in, y out, the cache read once and its new rows written; the
    # weights once
    return {"bytes": 2 * x + B * keys * (dc + dr) * 2 + M * ((dc + dr) * 2 + 12) +
                     2 * (HIDDEN * (dc + dr) + D_Q * HIDDEN + n_qcat * D_Q + HIDDEN * H * dc),
            "flops": 2 * M * HIDDEN * (dc + dr) + 2 * M * D_Q * (HIDDEN + n_qcat) +
                     B * tok * H * keys * (4 * dc + 2 * dr) + 2 * M * HIDDEN * H * dc}


def tolerance(case):
    """About four times the 2-norm error measured against 64 bits (rounding to
    bf16: 0.0017 for a projection, 0.0018 to 0.0027 where probabilities or a
    normalised latent are rounded too, 0.0035 at the end of a layer), and a
    bound on single values that allows several bf16 steps."""
    return {"append": {"rel": 7e-3, "max": 0.05},
            "query": {"rel": 1e-2, "max": 0.1},
            "attention": {"rel": 1e-2, "max": 0.1},
            "window": {"rel": 1e-2, "max": 0.1},
            "output": {"rel": 7e-3, "max": 0.05},
            "dense": {"rel": 1.1e-2, "max": 0.1},
            "layer": {"rel": 1.4e-2, "max": 0.1}}[case["op"]]


# -------------------------------------------------------------------- exact
def _rope(x, pos, d_r):
    """RoPE3D in 64 bits: x [..., n, d_r] (pairs last) at pos [n, 3]."""
    pairs, dims = ROPE[d_r]
    ang = []
    for axis in range(3):
        i = torch.arange(pairs[axis], device="cuda", dtype=torch.float64)
        ang.append(pos[:, axis].double()[:, None] * 10000.0 ** (-2.0 * i / dims[axis])[None])
    ang = torch.cat(ang, 1)
    cos, sin = ang.cos(), ang.sin()
    xp = x.reshape(*x.shape[:-1], d_r // 2, 2)
    return torch.stack([xp[..., 0] * cos - xp[..., 1] * sin,
                        xp[..., 0] * sin + xp[..., 1] * cos], -1).reshape(x.shape)


def _softmax_av(q, k, v):
    """softmax(q k^T / sqrt(d_h)) v for rows q, a block of rows at a time."""
    out = torch.empty(q.shape[0], v.shape[1], dtype=torch.float64, device="cuda")
    for r in range(0, q.shape[0], 8192):
        s = (q[r:r + 8192] @ k.T).mul_(HEAD_DIM ** -0.5)
        s.sub_(s.amax(1, keepdim=True)).exp_()
        out[r:r + 8192] = (s @ v) / s.sum(1, keepdim=True)
    return out


def _append(case, t, c, kr):
    """The cache once the chunk is in it; c and kr: what it held, in 64 bits."""
    T, W, S = _sizes(case)["T"], case["window"], case["sink"]
    cn = t["x"].double() @ t["w_dkv"].double().T
    cn = cn * (cn.square().mean(-1, keepdim=True) + EPS).rsqrt() * t["gamma"].double()
    kn = _rope(t["x"].double() @ t["w_kr"].double().T, t["pos"][0], case["d_r"])
    for i, f in enumerate(range(case["at"] - case["frames"], case["at"])):
        j = f if f < S else S + (f - S) % (W - S)
        c[:, j * T:(j + 1) * T] = cn[:, i * T:(i + 1) * T]
        kr[:, j * T:(j + 1) * T] = kn[:, i * T:(i + 1) * T]
    return c, kr


def _query(t):
    ct = t["x"].double() @ t["w_dq"].double().T
    return (ct * (ct.square().mean(-1, keepdim=True) + EPS).rsqrt()) @ t["w_qcat"].double().T


def _attend(case, q_c, q_r, q_pos, c, kr):
    """q_c [B, n, H, d_c], q_r unrotated; c, kr [B, keys, .] (kr rotated)."""
    B, n = q_c.shape[:2]
    out = torch.empty(B, n, HEADS, case["d_c"], dtype=torch.float64, device="cuda")
    for b in range(B):
        qr = _rope(q_r[b].double().transpose(0, 1), q_pos, case["d_r"]).transpose(0, 1)
        q = torch.cat([q_c[b].double(), qr], -1).reshape(n * HEADS, -1)
        k = torch.cat([c[b].double(), kr[b].double()], -1)
        out[b] = _softmax_av(q, k, c[b].double()).view(n, HEADS, -1)
    return out


def exact(case, seed):
    t = _inputs(case, seed)
    z = _sizes(case)
    op, B, dc = case["op"], case["batch"], case["d_c"]
    split = HEADS * dc
    if op == "append":
        c, kr = _append(case, t, t["c"].double(), t["kr"].double())
        return {"c": c, "kr": kr}
    if op == "query":
        q = _query(t)
        return {"q_c": q[..., :split].reshape(B, z["tok"], HEADS, dc),
                "q_r": q[..., split:].reshape(B, z["tok"], HEADS, case["d_r"])}
    if op == "output":
        return {"y": t["o_lat"].double().view(B, z["tok"], split) @ t["w_b"].double().T}
    n = z["keys"]
    if op == "attention":
        return {"o": _attend(case, t["q_c"], t["q_r"], t["pos"][0], t["c"][:, :n], t["kr"][:, :n])}
    if op == "window":
        # held frames are numbered in temporal order; keys and queries take
        # that number as their temporal coordinate
        slot_frames = _slot_frames(case)
        local = {f: i for i, f in enumerate(sorted(f for f in slot_frames if f >= 0))}
        times = [local[f] for f in slot_frames if f >= 0]
        kpos = torch.cat([torch.cat([torch.full((z["T"], 1), i, device="cuda", dtype=torch.int32),
                                     t["hw"]], 1) for i in times])
        qpos = t["pos"][0].clone()
        for f in range(case["at"] - case["frames"], case["at"]):
            qpos[t["pos"][0][:, 0] == f, 0] = local[f]
        kr = _rope(t["kr"][:, :n].double(), kpos, case["d_r"])
        return {"o": _attend(case, t["q_c"], t["q_r"], qpos, t["c"][:, :n], kr)}
    if op == "dense":
        c, kr = t["c"].double(), t["kr"].double()
        k = torch.cat([torch.einsum("bsc,hec->bhse", c, t["w_uk"].double()),
                       kr[:, None].expand(-1, HEADS, -1, -1)], -1)
        v = torch.einsum("bsc,hec->bhse", c, t["w_uv"].double())
        o = torch.empty(B, z["tok"], HEADS, HEAD_DIM, dtype=torch.float64, device="cuda")
        for b in range(B):
            for h in range(HEADS):
                o[b, :, h] = _softmax_av(t["q"][b, :, h].double(), k[b, h, :n], v[b, h, :n])
        return {"k": k, "v": v, "o": o}
    c, kr = _append(case, t, t["c"].double(), t["kr"].double())  # layer
    q = _query(t)
    o = _attend(case, q[..., :split].reshape(B, z["tok"], HEADS, dc),
                q[..., split:].reshape(B, z["tok"], HEADS, case["d_r"]), t["pos"][0], c[:, :n],
                kr[:, :n])
    return {"c": c, "kr": kr, "y": o.view(B, z["tok"], split) @ t["w_b"].double().T}
