"""Workloads of the METok hot path, as a program that serves long videos calls it.

Three kinds of case, one for each place where the path removes visual tokens:

  encode  after the vision encoder: event segmentation, text relevance, and the stage-1 compressor
          (key tokens + merge, or the paper's adaptive pooling), once per video;
  prune   during LLM prefill: text->visual attention scores, class-wise top-k and compaction of the
          hidden states, one level (`levels` 1, a call per pruning layer) or all three in one call;
  kv      before decoding: the per-layer K/V keep lists and the in-place compaction of the cache.

Sizes, ratios and head shapes are those of the configurations in `workloads.py` (8 to 512 frames of 16 to
196 tokens, the paper's 24-, 28- and 40-layer decoders); `draw` covers the ranges between them.  Inputs
are built on the GPU with the recipe of `workloads.py`: frames of an event share a base and differ by
noise, relevant events carry the text's direction, Q and K carry a rank-1 relevance.
"""

from __future__ import annotations

import math
import random

import torch

from paper_2506_02850_b200 import binding as B

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
BYTES = {"bf16": 2, "f32": 4}

# decoder shapes: query heads, K/V heads, head size, hidden width, layers
DECODERS = {"one": (1, 1, 64, 64, 1), "small": (14, 2, 64, 896, 24), "base": (28, 4, 128, 3584, 28),
            "large": (40, 40, 128, 5120, 40)}


def _encode(T, N, d, k, keep, dtype="bf16", mode="merge", fused=True, events="mixed", static=0.0, agg="mean",
            sim="flatten"):
    return {"kind": "encode", "dtype": dtype, "T": T, "N": N, "d": d, "k": k, "keep": keep, "mode": mode,
            "fused": fused, "events": events, "static": static, "agg": agg, "sim": sim}


def _prune(decoder, n_vis, Lt, r, levels=1, vis_start=0, dtype="bf16"):
    return {"kind": "prune", "dtype": dtype, "decoder": decoder, "n_vis": n_vis, "Lt": Lt, "r": r,
            "levels": levels, "vis_start": vis_start}


def _kv(decoder, n_vis, text, policy, ratio=1.0, l1=0, per_layer=False, vis_start=0, dtype="bf16"):
    return {"kind": "kv", "dtype": dtype, "decoder": decoder, "n_vis": n_vis, "text": text, "policy": policy,
            "ratio": ratio, "l1": l1, "per_layer": per_layer, "vis_start": vis_start}


def listed():
    return [
        # a clip of eight small frames in fp32: nothing but latency, launches and host work
        dict(_encode(8, 16, 64, 2, 0.5, dtype="f32"), name="encode_8x16_f32"),
        # a short video, 32 frames: the most common call of a chat server
        dict(_encode(32, 144, 1024, 4, 0.3), name="encode_32x144"),
        # the 128-frame video at the decoder's own width: the workload the benchmark is quoted on
        dict(_encode(128, 144, 3584, 16, 0.2), name="encode_128x144_wide"),
        # 512 frames cut into events of very different lengths, some background positions never changing
        dict(_encode(512, 144, 1024, 64, 0.2, events="zipf", static=0.05), name="encode_512x144"),
        # fp32 features of odd sizes: 61 frames of a 13 x 13 grid, a width that is not a multiple of 64
        dict(_encode(61, 169, 1156, 7, 0.25, dtype="f32"), name="encode_61x169_f32"),
        # the paper's own compressor (key frames, adaptive pooling) behind the separate segmentation call
        dict(_encode(64, 196, 1152, 8, 1.0, mode="pool", fused=False), name="pool_64x196"),
        # one pruning layer of the smallest decoder, 32 frames of 196 tokens, a short question
        dict(_prune("small", 6272, 24, 0.76), name="prune_small_6272"),
        # fp32 prefill with a system prompt before the video and odd sizes everywhere
        dict(_prune("small", 1999, 7, 0.55, vis_start=35, dtype="f32"), name="prune_small_1999_f32"),
        # the three pruning layers of the 7B decoder on the 128-frame video, in one call
        dict(_prune("base", 18432, 64, 0.5, levels=3), name="prune_base_18432_3levels"),
        # one pruning layer on the 512-frame video with a long question
        dict(_prune("base", 73728, 128, 0.5), name="prune_base_73728"),
        # 32 frames in the 7B decoder's cache, the paper's rule: visual rows leave every layer from l1 on
        dict(_kv("base", 6272, 80, "paper", l1=3), name="kv_base_6272_paper"),
        # the 128-frame video's cache, best-scored 6.5 % kept in all 28 layers
        dict(_kv("base", 18432, 64, "topk", ratio=0.065), name="kv_base_18432_topk"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_encode(rng):
    dtype = "f32" if rng.random() < 0.25 else "bf16"
    T = _log_int(rng, 4, 512)
    d = 8 * _log_int(rng, 8, 448)
    if dtype == "f32" and rng.random() < 0.5:
        d -= 4
    wide = dtype == "f32" and d > 2048                                   # rows the one-pass call does not take
    k = min(T, max(1, int(round(T / math.exp(rng.uniform(math.log(2), math.log(24)))))))
    agg = rng.choice(["mean", "max"])
    if rng.random() < 0.3:
        return _encode(T, rng.randint(4, 16) ** 2, d, k, 1.0, dtype, "pool", not wide and rng.random() < 0.5, "mixed", 0.0, agg,
                       "flatten")
    fused = not wide and rng.random() < 0.7
    sim = "flatten" if fused or rng.random() < 0.5 else "meanpool"
    return _encode(T, _log_int(rng, 16, 256), d, k, round(rng.uniform(0.1, 0.5), 3), dtype, "merge", fused,
                   rng.choice(["mixed", "zipf"]), rng.choice([0.0, 0.05]), agg, sim)


def _draw_prune(rng):
    f32 = rng.random() < 0.2
    decoder = rng.choice(["one", "small", "small", "base", "base", "base", "large"])
    return _prune(decoder, _log_int(rng, 64, 8192 if f32 else 73728), _log_int(rng, 1, 32 if f32 else 128),
                  round(rng.uniform(0.4, 0.8), 3), rng.choice([1, 1, 3]), rng.choice([0, rng.randint(1, 64)]),
                  "f32" if f32 else "bf16")


def _draw_kv(rng):
    policy = rng.choice(["topk", "topk", "paper", "given"])
    decoder = rng.choice(["one", "small", "base", "base", "large"])
    layers = DECODERS[decoder][4]
    return _kv(decoder, _log_int(rng, 64, 73728), _log_int(rng, 4, 256), policy,
               round(math.exp(rng.uniform(math.log(0.03), math.log(0.5))), 3), rng.randint(0, max(0, layers // 3)),
               policy == "topk" and rng.random() < 0.4, rng.choice([0, rng.randint(1, 64)]),
               "f32" if rng.random() < 0.15 else "bf16")


def _cost(case):
    """Work of a case in bytes of memory traffic: what keeps a drawn case below the largest listed one.
    fp32 contractions have no tensor-core form at full precision."""
    w = work(case)
    return w["bytes"] + w["flops"] / (4.0 if case["dtype"] == "f32" else 50.0)


def draw(rng: random.Random):
    most = max(_cost(c) for c in listed())
    while True:
        case = rng.choice([_draw_encode, _draw_encode, _draw_prune, _draw_prune, _draw_kv])(rng)
        if _cost(case) <= most and (case["kind"] != "kv" or _cache_bytes(case) <= 4.5e9):
            return case


# ---- inputs --------------------------------------------------------------------------------------


def _lengths(case):
    """Event lengths in frames: fixed by the case, their order by the seed."""
    T, k = case["T"], case["k"]
    if case["events"] == "zipf":
        h = sum(1.0 / i for i in range(1, k + 1))
        lens = [max(1, int(round(T / (i * h)))) for i in range(1, k + 1)]
    else:
        r = random.Random(1009 * T + k)
        w = [r.uniform(1.0, 8.0) for _ in range(k)]
        lens = [max(1, int(T * x / sum(w))) for x in w]
    while sum(lens) != T:
        i = lens.index(max(lens) if sum(lens) > T else min(lens))
        lens[i] += 1 if sum(lens) < T else -1
    return lens


def _ceil(x):
    return int(math.ceil(x - 1e-9))


def _prepare_encode(case, seed):
    T, N, d, k = case["T"], case["N"], case["d"], case["k"]
    dt = DTYPES[case["dtype"]]
    host = random.Random(seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    lens = _lengths(case)
    host.shuffle(lens)
    base = torch.randn((k, N, d), device="cuda", generator=g)
    live = torch.ones(N, 1, device="cuda")
    if case["static"] > 0:
        still = host.sample(range(N), max(1, int(round(case["static"] * N))))
        base[:, still, :] = torch.randn(d, device="cuda", generator=g)
        live[still] = 0.0
    w = torch.randn(d, device="cuda", generator=g)
    w /= w.norm()
    relevant = torch.zeros(k, 1, 1, device="cuda")
    relevant[host.sample(range(k), _ceil(0.5 * k))] = 1.0
    base += relevant * live * (0.25 * math.sqrt(d)) * w
    text = (3.0 * (w + 0.1 / math.sqrt(d) * torch.randn(d, device="cuda", generator=g))).to(dt)
    V = torch.empty((T, N, d), dtype=dt, device="cuda")
    f = 0
    for e, n in enumerate(lens):
        V[f:f + n] = base[e] + 0.1 * torch.randn((n, N, d), device="cuda", generator=g)
        f += n
    p = B.vision_params(0.5, case["keep"], case["keep"], event_agg=B.AGG_MAX if case["agg"] == "max" else B.AGG_MEAN,
                        mode=B.MODE_POOL if case["mode"] == "pool" else B.MODE_TOPK_MERGE)
    state = {"case": case, "V": V, "text": text, "params": p, "seg": None, "cv": None,
             "sim": B.SIM_MEANPOOL if case["sim"] == "meanpool" else B.SIM_FLATTEN}
    # a server keeps the result buffers of a video shape: made by a first call, zero where nothing is written
    _run_encode(state)
    for kept in (state["seg"], state["cv"]):
        for t in kept.values():
            if torch.is_tensor(t):
                t.zero_()
    return state


def _classes(case):
    """Tokens per frame, tokens of key events and of the others: the class of a token is that of its frame's
    event, so classes come in runs; the counts are fixed by the case, the order by the seed."""
    run = max(1, min(144, case["n_vis"] // 8))
    n_key = (case["n_vis"] // run + 1) // 2 * run
    return run, n_key, case["n_vis"] - n_key


def _prepare_prune(case, seed):
    Hq, Hkv, dh, D, _ = DECODERS[case["decoder"]]
    n_vis, Lt, v0 = case["n_vis"], case["Lt"], case["vis_start"]
    dt = DTYPES[case["dtype"]]
    host = random.Random(seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    run, n_key, n_rest = _classes(case)
    frames = [0] * (n_key // run) + [1] * (n_rest // run)
    host.shuffle(frames)
    classes = [c for f in frames for c in [f] * run]
    classes += [1] * (n_vis - len(classes))
    group = torch.tensor(classes, dtype=torch.int32, device="cuda")
    N0 = (n_key, n_rest)
    sizes = B.metok_prune_schedule_sizes(3, 0.5, case["r"], N0)
    q, kk, hid = [], [], []
    for s in range(case["levels"]):
        n = sizes[s]
        S = v0 + n + Lt
        Q = torch.randn((Hq, Lt, dh), device="cuda", generator=g) * dh ** -0.5
        K = torch.randn((Hkv, S, dh), device="cuda", generator=g) * dh ** -0.5
        rho = torch.randn(n, device="cuda", generator=g)
        if s == 0:
            rho += 0.5 - group.float()
        u = torch.randn((Hkv, 1, dh), device="cuda", generator=g)
        u *= math.sqrt(2.0 * math.sqrt(dh)) / u.norm(dim=-1, keepdim=True)
        K[:, v0:v0 + n] += rho[None, :, None] * u
        Q += u.repeat_interleave(Hq // Hkv, dim=0)
        q.append(Q.to(dt))
        kk.append(K.to(dt))
        hid.append(torch.randn((S, D), device="cuda", dtype=dt, generator=g))
    return {"case": case, "q": q, "k": kk, "hidden": hid, "group": group, "N0": N0, "sizes": sizes, "scale": dh ** -0.5}


def _cache_bytes(case):
    _, Hkv, dh, _, L = DECODERS[case["decoder"]]
    return 2.0 * L * Hkv * dh * (case["vis_start"] + case["n_vis"] + case["text"]) * BYTES[case["dtype"]]


def _prepare_kv(case, seed):
    _, Hkv, dh, _, L = DECODERS[case["decoder"]]
    n_vis = case["n_vis"]
    S = case["vis_start"] + n_vis + case["text"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    # one allocation holds the cache of all layers, a layer's K and V are views of it
    cache = torch.empty((L, 2, Hkv, S, dh), dtype=DTYPES[case["dtype"]], device="cuda").normal_(generator=g)
    state = {"case": case, "cache": cache, "S": S, "ks": [cache[l, 0] for l in range(L)],
             "vs": [cache[l, 1] for l in range(L)]}
    if case["policy"] == "topk":
        shape = (L, n_vis) if case["per_layer"] else (n_vis,)
        state["scores"] = torch.randn(shape, device="cuda", generator=g).exp() / n_vis
    if case["policy"] == "given":
        n = _kept(case)
        order = torch.rand((L, S), device="cuda", generator=g).argsort(dim=1)[:, :n].sort(dim=1).values
        lists = torch.zeros((L, S), dtype=torch.int32, device="cuda")
        lists[:, :n] = order.to(torch.int32)
        state["lists"] = lists
        state["lens"] = torch.full((L,), n, dtype=torch.int32, device="cuda")
    return state


def prepare(case, seed):
    return {"encode": _prepare_encode, "prune": _prepare_prune, "kv": _prepare_kv}[case["kind"]](case, seed)


# ---- one pass ------------------------------------------------------------------------------------


def _run_encode(s):
    if s["case"]["fused"]:
        seg = B.metok_segment_score_events(s["V"], s["case"]["k"], s["text"], out=s["seg"])
        cv = B.metok_compress_vision(s["V"], seg["event_offsets"], s["text"], s["params"], out=s["cv"], scored=seg)
    else:
        seg = B.metok_segment_events(s["V"], s["case"]["k"], s["sim"], out=s["seg"])
        cv = B.metok_compress_vision(s["V"], seg["event_offsets"], s["text"], s["params"], out=s["cv"])
    s["seg"], s["cv"] = seg, cv
    out = {n: seg[n] for n in ("sims", "boundaries", "event_offsets", "frame_event")}
    if s["case"]["fused"]:
        out["token_inv_norm"] = seg["token_inv_norm"]
    for n in ("out_feats", "out_src", "out_event", "out_members", "assign", "token_score", "frame_score",
              "event_score", "event_is_key", "n_out"):
        out[n] = cv[n]
    return out


def _run_prune(s):
    case = s["case"]
    if case["levels"] == 1:
        budgets = B.metok_retention_budgets(0.5, case["r"], 1, s["N0"])
        levels = [B.metok_prefill_prune(s["q"][0], s["k"][0], s["hidden"][0], case["vis_start"], case["n_vis"],
                                        s["group"], budgets, s["scale"])]
    else:
        levels = B.metok_prefill_prune_schedule(s["q"], s["k"], s["hidden"], case["vis_start"], s["group"], 0.5,
                                                case["r"], s["N0"], s["scale"])
    out = []
    for i, lv in enumerate(levels):
        n = case["vis_start"] + s["sizes"][i + 1] + case["Lt"]            # surviving rows, known to the host
        o = {"scores": lv["scores"], "S_out": lv["S_out"], "keep_idx": lv["keep_idx"][:n], "hidden": lv["hidden_out"][:n]}
        if case["levels"] > 1:
            o["origin"], o["group"] = lv["origin"], lv["token_group"]
        out.append(o)
    return out


def _kept(case):
    """Rows a compacted layer keeps."""
    rest = case["vis_start"] + case["text"]
    return rest if case["policy"] == "paper" else rest + min(case["n_vis"], _ceil(case["ratio"] * case["n_vis"]))


def _run_kv(s):
    case, cache = s["case"], s["cache"]
    args = (s["ks"], s["vs"], s["S"])
    span = (case["vis_start"], case["n_vis"])
    if case["policy"] == "topk":
        r = B.metok_kv_compact(*args, B.KV_TOPK, *span, keep_ratio=case["ratio"], scores=s["scores"])
    elif case["policy"] == "paper":
        r = B.metok_kv_compact(*args, B.KV_PAPER, *span, l1=case["l1"])
    else:
        r = B.metok_kv_compact(*args, B.KV_GIVEN, *span, keep_idx=s["lists"], keep_len=s["lens"])
    n = _kept(case)
    l1 = case["l1"] if case["policy"] == "paper" else 0                  # layers below l1 keep all their rows
    return {"keep_len": r["keep_len"], "new_len": r["new_len"], "lists_all": r["keep_idx"][:l1],
            "lists": r["keep_idx"][l1:, :n], "cache_all": cache[:l1], "cache": cache[l1:, :, :, :n]}


def run(state):
    return {"encode": _run_encode, "prune": _run_prune, "kv": _run_kv}[state["case"]["kind"]](state)


# ---- what a pass cannot do without ---------------------------------------------------------------


def work(case):
    b = BYTES[case["dtype"]]
    if case["kind"] == "encode":
        N, d, k = case["N"], case["d"], case["k"]
        tokens = case["T"] * N
        flops = 6.0 * tokens * d                                         # norms, frame and text products
        if case["mode"] == "merge":
            n_out = 0
            for n in _lengths(case):
                m = n * N
                keys = min(m, max(1, _ceil(case["keep"] * m)))
                n_out += keys
                flops += 2.0 * (m - keys) * keys * d + (m - keys) * d     # every other token against the keys, then the means
        else:
            side = int(round(math.sqrt(N)))
            windows = [(-(-side // s)) ** 2 for s in (2, 3, 4, 6)]
            n_out = case["T"] * sum(windows) / 4.0                       # half of the frames key frames, half of the events key events
            flops += tokens * d
        return {"bytes": (tokens + n_out) * d * b + tokens * (12.0 if case["fused"] else 8.0) + 12.0 * n_out, "flops": flops}
    if case["kind"] == "prune":
        Hq, Hkv, dh, D, _ = DECODERS[case["decoder"]]
        rest = case["vis_start"] + case["Lt"]
        _, n_key, n_rest = _classes(case)
        r = case["r"]
        sizes = [case["n_vis"], _ceil(r * n_key) + _ceil(0.5 * r * n_rest), _ceil(r * r * n_key), 0]
        nbytes = flops = 0.0
        for s in range(case["levels"]):
            S, out = sizes[s] + rest, sizes[s + 1] + rest
            nbytes += (Hq * case["Lt"] + Hkv * S) * dh * b + 2.0 * out * D * b + 8.0 * sizes[s] + 4.0 * out
            flops += 2.0 * Hq * case["Lt"] * S * dh
        return {"bytes": nbytes, "flops": flops}
    _, Hkv, dh, _, L = DECODERS[case["decoder"]]
    n = _kept(case)
    S = case["vis_start"] + case["n_vis"] + case["text"]
    l1 = case["l1"] if case["policy"] == "paper" else 0
    moved = max(0, n - case["vis_start"])                                # rows before the visual span stay where they are
    scores = 4.0 * case["n_vis"] * (L if case["per_layer"] else 1) if case["policy"] == "topk" else 0.0
    return {"bytes": (L - l1) * (2.0 * 2.0 * Hkv * moved * dh * b + 4.0 * n) + 4.0 * l1 * S + scores, "flops": 0.0}


def tolerance(case):
    """kv moves rows: exact.  prune: fp32 scores, then rows moved unchanged.  encode: fp32 scores; averaged features
    rounded to the input's type; tokens between two equally similar keys may join either."""
    if case["kind"] == "kv":
        return "exact"
    if case["kind"] == "prune" or case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4, "differ": 1e-3}
    return {"rel": 1e-2, "max": 0.4, "differ": 5e-3}
