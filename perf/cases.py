"""The work a program built on this library has it do, as cases that can be timed.

A program that streams a world model calls the library per generated chunk: it looks up stored chunks by camera pose
(`retrieve`), attends over window and retrieved chunks once per layer and denoising step (`attention`), and stores the
chunk that leaves the window (`store`: score, select and gather all layers in one call).  `step` is that whole loop.
The other kinds are the options of the same path: per-head keep-sets (`heads`), ranking stored chunks by the current
query (`query`), and pose retrieval over large candidate arrays (`scan`).

Sizes are those of wkinputs/workloads.py (Matrix-Game shape: 12 heads x 880 tokens per frame; LingBot shape: 40 heads x
1,560), whose token counts are multiples of neither 64 nor 128.  Keys follow the same recipe as wkinputs: a base vector
per position, 30 % of the positions redrawn per frame, per-frame noise; queries and values are unit normals; poses are
jittered loops that revisit their start, or random.
"""
import math

import numpy as np
import torch

from paper_2605_22718_b200 import SCORE_PER_HEAD, WorldKV

DEV = "cuda:0"
BF = torch.bfloat16


def listed():
    return [
        # the smallest attention call: one frame of queries, two heads, one retrieved chunk (workload cfg0)
        dict(name="attention_tiny", kind="attention", heads=2, T=880, q_frames=1, window=2, segs=1, slots=8, k=1, keep=440),
        # an ordinary call: the paper's own window (sink 3 + recent 3 frames as two segments, six retrieved chunks)
        dict(name="attention_mg", kind="attention", heads=12, T=880, q_frames=3, window=6, segs=2, slots=32, k=6, keep=440),
        # the larger model: 40 heads, 4,680 queries, top-8 (workload cfg3)
        dict(name="attention_lb", kind="attention", heads=40, T=1560, q_frames=3, window=6, segs=1, slots=12, k=8, keep=780),
        # a whole minute of compressed history attended at once (workload cfg4c)
        dict(name="attention_history", kind="attention", heads=12, T=880, q_frames=3, window=0, segs=0, slots=125, k=125,
             keep=440),
        # one chunk step of the full denoising pass: retrieve, 30 layers x 4 steps of attention, store (workload cfg2 with
        # a shorter pool)
        dict(name="step_mg", kind="step", layers=30, steps=4, heads=12, T=880, window=6, slots=16, k=8, keep=440),
        # storing the chunk that leaves the window, all layers in one call, on both model shapes
        dict(name="store_mg", kind="store", layers=30, heads=12, T=880, slots=3, keep=440),
        dict(name="store_lb", kind="store", layers=40, heads=40, T=1560, slots=2, keep=780),
        # keep-sets per head instead of per token
        dict(name="heads_mg", kind="heads", layers=30, heads=12, T=880, keep=440),
        # the latency-bound call in front of every step: a two-minute pool, top-8
        dict(name="retrieve_pool", kind="retrieve", slots=250, k=8, loop=True),
        # pose retrieval over large candidate sets
        dict(name="scan_1m", kind="scan", n=1 << 20, k=16, masked=False),
        dict(name="scan_16m", kind="scan", n=1 << 24, k=16, masked=False),
        # ranking a two-minute pool by the attention the current query pays each chunk
        dict(name="query_mg", kind="query", heads=12, T=880, lq=2640, slots=250, k=4, keep=440),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["attention", "attention", "attention", "step", "store", "store", "heads", "retrieve", "scan", "query"])
    heads = rng.choice([1, 2, 5, 8, 12, 12, 16, 24, 40])
    T = _log(rng, 96, 1560)
    # retained non-anchor tokens: the retention ladder, or any number
    keep = max(1, rng.choice([T // 4, T // 2, T // 2, T, rng.randint(1, 2 * T - 1)]))
    if kind == "attention":
        k = rng.choice([0, 1, 2, 4, 6, 8, 16, 16, 60, 125])
        if k > 16:                       # a whole history: the smaller model's shape at most
            heads, T, keep = min(heads, 12), min(T, 880), min(keep, T // 2)
            keep = max(1, min(keep, T))
        window = rng.randint(0, 6) if k else rng.randint(1, 6)
        return dict(kind=kind, heads=heads, T=T, q_frames=rng.choice([1, 3, 3]), window=window,
                    segs=min(window, rng.choice([1, 1, 2, 3])), slots=k + rng.randint(1, 8), k=k, keep=keep)
    if kind == "step":
        heads, T = min(heads, 12), min(T, 880)
        return dict(kind=kind, layers=rng.randint(2, 30), steps=rng.choice([1, 2, 4]), heads=heads, T=T,
                    window=rng.choice([3, 6]), slots=rng.randint(9, 16), k=rng.randint(1, 8), keep=max(1, T // 2))
    if kind in ("store", "heads"):
        layers = _log(rng, 1, 40)
        c = dict(kind=kind, layers=layers, heads=heads, T=T, keep=min(keep, 2 * T - 1))
        if kind == "store":
            c["slots"] = rng.randint(2, 3)
        return c
    if kind == "retrieve":
        return dict(kind=kind, slots=_log(rng, 8, 1024), k=rng.randint(1, 16), loop=rng.random() < 0.5)
    if kind == "scan":
        return dict(kind=kind, n=_log(rng, 1 << 14, 1 << 24), k=rng.choice([1, 4, 16, 16, 64]), masked=rng.random() < 0.3)
    return dict(kind=kind, heads=min(heads, 12), T=min(T, 880), lq=_log(rng, 128, 2640), slots=_log(rng, 8, 250), k=4,
                keep=max(1, min(T, 880) // 2))


# ------------------------------------------------------------------------------------------------ inputs
def _normal(gen, *shape):
    return torch.randn(shape, generator=gen, device=DEV, dtype=torch.float32).to(BF)


def _keys(gen, layers, T, D, frames=3, sigma=0.1):
    """[layers, frames * T, D]: a base vector per position, 30 % of the positions redrawn per frame, plus frame noise."""
    out = torch.empty((layers, frames * T, D), dtype=BF, device=DEV)
    base = torch.randn((layers, T, D), generator=gen, device=DEV)
    for f in range(frames):
        if f:
            redrawn = torch.rand((layers, T, 1), generator=gen, device=DEV) < 0.3
            base = torch.where(redrawn, torch.randn((layers, T, D), generator=gen, device=DEV), base)
        out[:, f * T:(f + 1) * T] = base + sigma * torch.randn((layers, T, D), generator=gen, device=DEV)
    return out


def _poses(seed, n, loop):
    """[n, 8] fp32: translation, 0, unit quaternion; a jittered circle walked once around, or random poses."""
    rng = np.random.default_rng([seed, n])
    if loop:
        phi = 2 * np.pi * np.arange(n) / n
        t = np.stack([10 * np.cos(phi), 10 * np.sin(phi), np.zeros(n)], -1) + 0.01 * rng.standard_normal((n, 3))
        yaw = phi + np.pi / 2 + 0.01 * rng.standard_normal(n)
        pitch = 0.01 * rng.standard_normal(n)
        cy, sy, cp, sp = np.cos(yaw / 2), np.sin(yaw / 2), np.cos(pitch / 2), np.sin(pitch / 2)
        q = np.stack([cy * cp, -sy * sp, cy * sp, sy * cp], -1)
    else:
        t, q = rng.standard_normal((n, 3)), rng.standard_normal((n, 4))
    out = np.zeros((n, 8), dtype=np.float32)
    out[:, :3] = t
    out[:, 4:] = q / np.linalg.norm(q, axis=1, keepdims=True)
    return out


def _fill(kv, gen, layers, T, D, count, poses):
    """Stores `count` chunks the way a program does: one call per chunk for all layers."""
    for c in range(count):
        kv.pool_compress_append(0, layers, _keys(gen, layers, T, D), _normal(gen, layers, 3 * T, D), poses[c], chunk_tag=c)


def _stored_rows(kv, layers, slots, D):
    """Views of every slot's stored rows in the pool buffer: per slot (K [layers, C, D], V [layers, C, D])."""
    n = layers * slots * kv.C * D * 2
    pitch = (n + 255) // 256 * 256
    K = kv.pool[:n].view(BF).view(layers, slots, kv.C, D)
    V = kv.pool[pitch:pitch + n].view(BF).view(layers, slots, kv.C, D)
    return [(K[:, s], V[:, s]) for s in range(slots)]


def _pick_slots(seed, slots, k):
    """Slot ids as retrieval returns them: distinct, in no particular order."""
    perm = np.random.default_rng([seed, 7]).permutation(slots)[:max(k, 1)]
    return torch.tensor(perm.astype(np.int32), device=DEV)


# ------------------------------------------------------------------------------------------------ preparation
def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    return {"attention": _prep_attention, "step": _prep_step, "store": _prep_store, "heads": _prep_store,
            "retrieve": _prep_retrieve, "scan": _prep_scan, "query": _prep_query}[case["kind"]](case, seed, gen)


def _prep_attention(c, seed, gen):
    H, T, D = c["heads"], c["T"], c["heads"] * 128
    lq = c["q_frames"] * T
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=T, n_keep=c["keep"], pool_slots=c["slots"], max_k=max(1, c["k"]),
                 max_dense_segments=4, max_batch=1, max_lq=lq)
    _fill(kv, gen, 1, T, D, c["slots"], _poses(seed, c["slots"], True))
    segs = [(_keys(gen, 1, T, D, c["q_frames"]).view(lq, H, 128), _normal(gen, lq, H, 128))]
    if c["window"]:
        n = c["window"] * T
        K, V = _keys(gen, 1, T, D, c["window"]).view(n, H, 128), _normal(gen, n, H, 128)
        cut = [n * i // c["segs"] for i in range(c["segs"] + 1)]
        segs += [(K[a:b], V[a:b]) for a, b in zip(cut, cut[1:])]
    return dict(kind="attention", kv=kv, Q=_normal(gen, lq, H, 128), segs=segs, slots=_pick_slots(seed, c["slots"], c["k"]),
                k=c["k"], O=torch.empty((lq, H, 128), dtype=BF, device=DEV),
                lse=torch.empty((H, lq), dtype=torch.float32, device=DEV))


def _prep_step(c, seed, gen):
    L, S, H, T, D = c["layers"], c["steps"], c["heads"], c["T"], c["heads"] * 128
    lq, nw = 3 * T, c["window"] * T
    kv = WorldKV(n_layers=L, n_heads=H, tokens_per_frame=T, n_keep=c["keep"], pool_slots=c["slots"], max_k=c["k"],
                 max_dense_segments=2, max_batch=L, max_lq=lq)
    poses = _poses(seed, c["slots"] + 64, True)
    _fill(kv, gen, L, T, D, c["slots"], poses)
    return dict(kind="step", kv=kv, layers=L, steps=S, k=c["k"], poses=poses[c["slots"]:], at=0,
                Q=_normal(gen, L, S, lq, H, 128), O=torch.empty((L, S, lq, H, 128), dtype=BF, device=DEV),
                curK=_keys(gen, L, T, D).view(L, lq, H, 128), curV=_normal(gen, L, lq, H, 128),
                winK=_keys(gen, L, T, D, c["window"]).view(L, nw, H, 128), winV=_normal(gen, L, nw, H, 128),
                oldK=_keys(gen, L, T, D), oldV=_normal(gen, L, 3 * T, D), rows=_stored_rows(kv, L, c["slots"], D),
                slots=torch.empty((max(1, c["k"]),), dtype=torch.int32, device=DEV),
                keep=torch.empty((L, kv.C), dtype=torch.int32, device=DEV))


def _prep_store(c, seed, gen):
    L, H, T, D = c["layers"], c["heads"], c["T"], c["heads"] * 128
    per_head = c["kind"] == "heads"
    slots = c.get("slots", 1)
    kv = WorldKV(n_layers=L, n_heads=H, tokens_per_frame=T, n_keep=c["keep"], pool_slots=slots, max_k=1, max_batch=L,
                 max_lq=1, score_mode=SCORE_PER_HEAD if per_head else 0)
    s = dict(kind=c["kind"], kv=kv, layers=L, K=_keys(gen, L, T, D), at=0,
             keep=torch.empty((L, H, kv.C) if per_head else (L, kv.C), dtype=torch.int32, device=DEV))
    if not per_head:
        s["V"] = _normal(gen, L, 3 * T, D)
        s["poses"] = _poses(seed, 64, True)
        s["rows"] = _stored_rows(kv, L, slots, D)
        for i in range(slots):          # a running program's pool is full: every further chunk replaces the oldest
            kv.pool_compress_append(0, L, s["K"], s["V"], s["poses"][i], chunk_tag=i, keep_idx=s["keep"])
    return s


def _prep_retrieve(c, seed, gen):
    # the stored rows do not matter to pose retrieval: a small row shape keeps the pool small
    kv = WorldKV(n_layers=1, n_heads=1, tokens_per_frame=8, n_keep=4, pool_slots=c["slots"], max_k=c["k"], max_lq=1)
    poses = _poses(seed, c["slots"] + 32, c["loop"])
    K, V = _keys(gen, 1, 8, 128), _normal(gen, 1, 24, 128)
    for i in range(c["slots"]):
        kv.pool_compress_append(0, 1, K, V, poses[i], chunk_tag=i)
    return dict(kind="retrieve", kv=kv, poses=poses[c["slots"]:], at=0, k=c["k"],
                slots=torch.empty((c["k"],), dtype=torch.int32, device=DEV),
                dist=torch.empty((c["k"],), dtype=torch.float64, device=DEV))


def _prep_scan(c, seed, gen):
    n = c["n"]
    kv = WorldKV(n_layers=1, n_heads=1, tokens_per_frame=8, n_keep=4, pool_slots=1, max_k=1, max_lq=1)
    poses = torch.zeros((n, 8), dtype=torch.float32, device=DEV)
    poses[:, :3] = torch.randn((n, 3), generator=gen, device=DEV)
    q = torch.randn((n, 4), generator=gen, device=DEV)
    poses[:, 4:] = q / q.norm(dim=1, keepdim=True)
    valid = (torch.rand(n, generator=gen, device=DEV) < 0.9).to(torch.int32) if c["masked"] else None
    return dict(kind="scan", kv=kv, poses=poses, valid=valid, cur=_poses(seed, 32, False), at=0, k=c["k"],
                ids=torch.empty((c["k"],), dtype=torch.int32, device=DEV),
                dist=torch.empty((c["k"],), dtype=torch.float64, device=DEV),
                scratch=torch.empty(kv.lib.wk_retrieve_scan_scratch_bytes(), dtype=torch.uint8, device=DEV))


def _prep_query(c, seed, gen):
    H, T, D, lq = c["heads"], c["T"], c["heads"] * 128, c["lq"]
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=T, n_keep=c["keep"], pool_slots=c["slots"], max_k=c["k"],
                 max_batch=1, max_lq=lq)
    _fill(kv, gen, 1, T, D, c["slots"], _poses(seed, c["slots"], True))
    # The current view shows places seen before: shares of the queries look for keys of k stored chunks (4 : 3 : 2 : 1 of
    # half of the rows), the other half looks for nothing in particular.
    Q = _normal(gen, lq, H, 128)
    rows = _stored_rows(kv, 1, c["slots"], D)
    at = 0
    for rank, s in enumerate(np.random.default_rng([seed, 9]).permutation(c["slots"])[:c["k"]]):
        n = min(kv.C, max(1, lq * (c["k"] - rank) // (c["k"] * (c["k"] + 1))))
        pick = torch.randperm(kv.C, generator=gen, device=DEV)[:n]
        Q[at:at + n] = (1.5 * rows[int(s)][0][0, pick].float()).to(BF).view(n, H, 128)
        at += n
    return dict(kind="query", kv=kv, Q=Q, k=c["k"], slots=torch.empty((c["k"],), dtype=torch.int32, device=DEV),
                score=torch.empty((c["k"],), dtype=torch.float32, device=DEV))


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    kv, kind = s["kv"], s["kind"]
    if kind == "attention":
        kv.memory_attention(0, s["Q"], s["segs"], s["slots"], s["k"], O=s["O"], lse_out=s["lse"])
        return s["O"], s["lse"]
    if kind == "query":
        kv.retrieve_query(0, s["Q"], s["k"], slots_out=s["slots"], score_out=s["score"])
        return s["slots"], s["score"]
    if kind == "heads":
        return kv.compress_chunk(s["K"], keep_idx_out=s["keep"])
    at = s["at"]
    s["at"] = at + 1
    if kind == "scan":
        kv.retrieve_scan(s["poses"], s["cur"][at % len(s["cur"])], s["k"], valid=s["valid"], ids_out=s["ids"],
                         dist_out=s["dist"], scratch=s["scratch"])
        return s["ids"], s["dist"]
    pose = s["poses"][at % len(s["poses"])]
    if kind == "retrieve":
        kv.retrieve(pose, s["k"], slots_out=s["slots"], dist_out=s["dist"])
        return s["slots"], s["dist"]
    if kind == "store":
        slot, _, keep = kv.pool_compress_append(0, s["layers"], s["K"], s["V"], pose, chunk_tag=at,
                                                evict_oldest_if_full=True, keep_idx=s["keep"])
        return keep, s["rows"][slot]
    _, n = kv.retrieve(pose, s["k"], slots_out=s["slots"])
    for t in range(s["steps"]):
        for l in range(s["layers"]):
            kv.memory_attention(l, s["Q"][l, t], [(s["curK"][l], s["curV"][l]), (s["winK"][l], s["winV"][l])], s["slots"], n,
                                O=s["O"][l, t])
    slot, _, keep = kv.pool_compress_append(0, s["layers"], s["oldK"], s["oldV"], pose, chunk_tag=at,
                                            evict_oldest_if_full=True, keep_idx=s["keep"])
    return s["O"], s["slots"], keep, s["rows"][slot]


# ------------------------------------------------------------------------------------------------ work and tolerance
def _attention_work(heads, lq, lkv):
    row = heads * 128 * 2
    return 2 * lq * row + 2 * lkv * row, 4.0 * lq * lkv * 128 * heads


def _store_bytes(layers, heads, T, keep):
    row = heads * 128 * 2
    # every key once, the kept rows of V once, the kept rows of both written once, the index list written
    return layers * (3 * T * row + 3 * (T + keep) * row + 4 * (T + keep))


def work(case):
    c, kind = case, case["kind"]
    if kind == "attention":
        lq = c["q_frames"] * c["T"]
        b, f = _attention_work(c["heads"], lq, lq + c["window"] * c["T"] + c["k"] * (c["T"] + c["keep"]))
        return {"bytes": b + 4 * c["heads"] * lq, "flops": f}
    if kind == "step":
        lq = 3 * c["T"]
        b, f = _attention_work(c["heads"], lq, lq + c["window"] * c["T"] + c["k"] * (c["T"] + c["keep"]))
        n = c["layers"] * c["steps"]
        return {"bytes": n * b + _store_bytes(c["layers"], c["heads"], c["T"], c["keep"]), "flops": n * f}
    if kind == "store":
        return {"bytes": _store_bytes(c["layers"], c["heads"], c["T"], c["keep"]),
                "flops": 4.0 * c["layers"] * 3 * c["T"] * c["heads"] * 128}
    if kind == "heads":
        n = c["layers"] * c["heads"]
        return {"bytes": n * (3 * c["T"] * 256 + 4 * (c["T"] + c["keep"])), "flops": 4.0 * n * 3 * c["T"] * 128}
    if kind == "retrieve":
        return {"bytes": 36 * c["slots"] + 12 * c["k"], "flops": 30.0 * c["slots"]}
    if kind == "scan":
        return {"bytes": (36 if c["masked"] else 32) * c["n"] + 12 * c["k"], "flops": 30.0 * c["n"]}
    rows = c["slots"] * (c["T"] + c["keep"])
    return {"bytes": (rows + c["lq"]) * c["heads"] * 256 + 8 * c["k"], "flops": 2.0 * c["lq"] * rows * 128 * c["heads"]}


def tolerance(case):
    """Four times what the path was measured to differ by from the same computation in 64 bits (80 bits for the distances)."""
    kind = case["kind"]
    if kind in ("attention", "step"):
        # P and the output are rounded to bf16: measured rel 2.3e-3, largest difference 1.1e-2 of the value or the rms
        return {"rel": 9e-3, "max": 0.045}
    if kind == "query":
        # fp32 sums over fp32 log-sum-exps: measured 4e-7 on these few scores, 1e-5 is what 32-bit sums of this length give
        return {"rel": 1e-5, "max": 4e-5}
    if kind in ("retrieve", "scan"):
        # fp64 distances; acos near 1 loses a few digits: measured rel 4e-14, largest 7e-13 (a revisited pose)
        return {"rel": 2e-13, "max": 3e-12}
    return "exact"            # indices and copied rows
