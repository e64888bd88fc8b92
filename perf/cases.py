"""Performance cases of the serving path, each through the public Python entry points.

Four kinds of work, with the sizes of this repository's workloads (the benchmark's decode, prefill, router,
K-means and full-forward workloads and the tiny layer of the tests) and sizes between them:

  route    queries -> expert ids (``route``; ``route_top2`` where the caller wants the margin too)
  layer    route + batch plan + routed LoRA projections, grouped as a decoder block issues them
  kmeans   one Lloyd iteration: assign, group, update
  forward  full decoder forward of packed requests, adapters on all seven projections of every block

A case is a dict of plain values; `prepare` turns it and a seed into what a serving process holds (weights,
adapter pools, centroid table, buffers) plus one batch of inputs, `run` is one pass over that batch.
"""
import math
import random

import numpy as np
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin

DEV = "cuda"
SCALE = 2.0
# projections that a decoder block issues together, as indices into the seven of mi.TINYLLAMA_PROJECTIONS
BLOCK_GROUPS = ((0, 1, 2), (3,), (4, 5), (6,))
MODEL_SLOTS = 128   # adapters of a decoder's pools that are resident on the GPU


def listed():
    return [
        # one request arrives and is routed over the 5 000 topics of the paper's larger table
        {"name": "route_one_request", "kind": "route", "Q": 1, "K": 5000, "D": 768, "want": "sim"},
        # a corpus is routed offline against the full topic table (the benchmark's router workload)
        {"name": "route_corpus", "kind": "route", "Q": 65536, "K": 5000, "D": 768, "want": "id"},
        # the tests' tiny layer: 16 ragged requests through one 256 -> 256 projection, rank 8
        {"name": "layer_tiny", "kind": "layer", "shape": "one", "d_in": 256, "d_out": 256, "R": 16, "lo": 1, "hi": 32,
         "K": 8, "D": 64, "E": 8, "r": 8, "kept": 1.0, "adaptive": False},
        # a decode step of a lightly loaded server: 24 running requests, one token each
        {"name": "decode_24", "kind": "layer", "shape": "block", "R": 24, "lo": 1, "hi": 1, "K": 500, "D": 768,
         "E": 500, "r": 64, "kept": 1.0, "adaptive": False},
        # a decode step of a busy server (the benchmark's default workload)
        {"name": "decode_256", "kind": "layer", "shape": "block", "R": 256, "lo": 1, "hi": 1, "K": 500, "D": 768,
         "E": 500, "r": 64, "kept": 1.0, "adaptive": False},
        # decode at the paper's rank with 387 of 500 topics retained and a rank per topic; odd batch
        {"name": "decode_rank128", "kind": "layer", "shape": "block", "R": 187, "lo": 1, "hi": 1, "K": 500, "D": 768,
         "E": 500, "r": 128, "kept": 0.774, "adaptive": True},
        # prompts of equal length, skewed experts (the benchmark's prefill workload)
        {"name": "prefill_32x512", "kind": "layer", "shape": "block", "R": 32, "lo": 512, "hi": 512, "K": 5000,
         "D": 768, "E": 5000, "r": 16, "kept": 1.0, "adaptive": False},
        # a few ragged prompts, some of them on topics without an adapter
        {"name": "prefill_ragged", "kind": "layer", "shape": "block", "R": 9, "lo": 65, "hi": 700, "K": 500, "D": 768,
         "E": 500, "r": 64, "kept": 0.774, "adaptive": False},
        # one iteration of the topic model over document embeddings
        {"name": "kmeans_40000", "kind": "kmeans", "N": 40000, "K": 1000, "D": 768},
        # perplexity evaluation: all-position logits (the benchmark's full-forward workload)
        {"name": "forward_64x256", "kind": "forward", "R": 64, "lo": 256, "hi": 256, "r": 64, "logits": "all",
         "base": "bf16"},
        # ragged prompts entering generation: only the last position's logits are wanted
        {"name": "forward_ragged", "kind": "forward", "R": 11, "lo": 65, "hi": 600, "r": 64, "logits": "last",
         "base": "bf16"},
        # a handful of short queries on the 8-bit base
        {"name": "forward_short_fp8", "kind": "forward", "R": 6, "lo": 3, "hi": 40, "r": 16, "logits": "last",
         "base": "fp8"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["route", "decode", "decode", "prefill", "prefill", "tiny", "kmeans", "forward", "forward"])
    D = rng.choice([64, 384, 768, 8 * rng.randint(8, 96)])
    if kind == "route":
        return {"kind": "route", "Q": _log_int(rng, 1, 65536), "K": _log_int(rng, 8, 5000), "D": D,
                "want": rng.choice(["id", "id", "sim", "top2"])}
    if kind == "kmeans":
        return {"kind": "kmeans", "N": _log_int(rng, 2000, 65536), "K": _log_int(rng, 20, 1000), "D": D}
    if kind == "tiny":
        return {"kind": "layer", "shape": "one", "d_in": 64 * rng.randint(1, 12), "d_out": 8 * rng.randint(4, 96),
                "R": rng.randint(2, 40), "lo": 1, "hi": rng.randint(2, 40), "K": 16, "D": D, "E": 16,
                "r": 8 * rng.randint(1, 4), "kept": rng.choice([1.0, 0.8]), "adaptive": False}
    if kind == "decode":
        r = rng.choice([8, 16, 32, 64, 64, 128, 8 * rng.randint(1, 16)])
        return {"kind": "layer", "shape": "block", "R": _log_int(rng, 1, 400), "lo": 1, "hi": 1,
                "K": rng.choice([500, 5000]), "D": 768, "E": rng.choice([100, 500]), "r": r,
                "kept": rng.choice([1.0, 0.774]), "adaptive": rng.random() < 0.3}
    if kind == "prefill":
        lo = rng.randint(64, 300)
        hi = rng.randint(lo, 700)
        R = _log_int(rng, 2, max(2, 16384 // hi))
        r = rng.choice([8, 16, 32, 64, 8 * rng.randint(1, 16)])
        return {"kind": "layer", "shape": "block", "R": R, "lo": lo, "hi": hi, "K": 500, "D": 768, "E": 500, "r": r,
                "kept": rng.choice([1.0, 0.774]), "adaptive": rng.random() < 0.3}
    lo = rng.choice([rng.randint(1, 24), rng.randint(64, 256)])
    hi = rng.randint(lo, 48 if lo < 64 else 600)
    return {"kind": "forward", "R": _log_int(rng, 2, min(64, max(2, 16384 // hi))), "lo": lo, "hi": hi,
            "r": rng.choice([8, 16, 32, 64, 64, 8 * rng.randint(1, 8)]), "logits": rng.choice(["all", "last", "last"]),
            "base": rng.choice(["bf16", "bf16", "fp8"])}


# ------------------------------------------------------------------ sizes that follow from a case

def _lengths(case):
    """Request lengths: part of the case (they decide the work), not of the seed."""
    if case["lo"] == case["hi"]:
        return [case["lo"]] * case["R"]
    rng = random.Random(case["R"] * 1000003 + case["lo"] * 1009 + case["hi"])
    return [rng.randint(case["lo"], case["hi"]) for _ in range(case["R"])]


def _projections(case):
    return (("p", case["d_in"], case["d_out"]),) if case["shape"] == "one" else mi.TINYLLAMA_PROJECTIONS


def _distinct(draws, of):
    """Expected number of distinct values in `draws` uniform draws out of `of`."""
    return of * (1.0 - (1.0 - 1.0 / of) ** draws)


def work(case):
    kind = case["kind"]
    if kind == "route":
        Q, K, D = case["Q"], case["K"], case["D"]
        return {"bytes": (Q + K) * D * 2 + Q * 4, "flops": 2.0 * Q * K * D}
    if kind == "kmeans":
        N, K, D = case["N"], case["K"], case["D"]
        return {"bytes": (N + 2 * K) * D * 2 + N * 4, "flops": 2.0 * N * K * D}
    T, R, r = sum(_lengths(case)), case["R"], case["r"]
    if kind == "layer":
        kept = case["kept"]
        r_mean = r * (0.5625 if case["adaptive"] else 1.0)   # ranks r/8, r/4, ... r in equal shares
        ids = _distinct(R, case["E"]) * kept
        b = (R + case["K"]) * case["D"] * 2.0
        f = 2.0 * R * case["K"] * case["D"]
        for _, di, do in _projections(case):
            b += 2.0 * (do * di + T * (di + do)) + ids * r_mean * (di + do) * 2
            f += 2.0 * T * di * do + 2.0 * T * kept * r_mean * (di + do)
        return {"bytes": b, "flops": f}
    cfg = mi.DecoderConfig()
    ids = _distinct(R, MODEL_SLOTS)
    wb = 1.0 if case["base"] == "fp8" else 2.0
    b, f = T * cfg.hidden * 2.0, 0.0
    for _, di, do in cfg.projections():
        b += cfg.n_layers * (wb * do * di + ids * r * (di + do) * 2)
        f += cfg.n_layers * (2.0 * T * di * do + 2.0 * T * r * (di + do))
    f += cfg.n_layers * sum(2.0 * n * (n + 1) * cfg.n_heads * cfg.head_dim for n in _lengths(case))   # causal attention
    rows = T if case["logits"] == "all" else R
    b += 2.0 * cfg.vocab * cfg.hidden + 2.0 * rows * cfg.vocab
    f += 2.0 * rows * cfg.vocab * cfg.hidden
    return {"bytes": b, "flops": f}


def tolerance(case):
    # Measured with the same inputs through the other kernel family (other summation orders) and through 64-bit
    # arithmetic; about four times what was seen.
    if case["kind"] == "route":      # ids bit-equal away from ties; similarities and margins are 32-bit sums
        return {"rel": 1e-4, "max": 1e-2, "differ": 1e-3}
    if case["kind"] == "kmeans":     # means rounded once to bf16
        return {"rel": 5e-3, "max": 2e-2, "differ": 1e-3}
    if case["kind"] == "layer":      # one bf16 rounding of 32-bit sums
        return {"rel": 5e-3, "max": 2e-2, "differ": 1e-3}
    # 22 blocks of chained bf16 storage: the two kernel families differ by 2.1e-2 (8e-3 for a short batch), each of
    # them from 64-bit arithmetic by about as much
    return {"rel": 3e-2, "max": 5e-1, "differ": 0.0}


# ------------------------------------------------------------------ inputs

def _seed(seed, *stream):
    return mi._mix(int(seed), *stream)


def _normal(shape, std, seed, *stream):
    return mi.normal_bf16(shape, std, seed, *stream, device=DEV)


def _pool(case_E, slots, r, d_in, d_out, slot_of_expert, slot_rank, seed, *stream):
    A = _normal((slots, r, d_in), 0.02, seed, *stream, 1)
    B = _normal((slots, d_out, r), 0.02, seed, *stream, 2)
    return moin.Pool(A, B, slot_of_expert, slot_rank=slot_rank)


def _prepare_route(case, seed):
    rc = mi.planted_router(case["K"], case["Q"], case["D"], seed, device=DEV)
    return {"router": moin.Router(rc.centroids), "queries": rc.queries,
            "expert": torch.empty(case["Q"], dtype=torch.int32, device=DEV),
            "sim": torch.empty(case["Q"], dtype=torch.float32, device=DEV) if case["want"] == "sim" else None}


def _run_route(case, s):
    if case["want"] == "top2":
        return moin.route_top2(s["router"], s["queries"])
    moin.route(s["router"], s["queries"], out_expert=s["expert"], out_best_sim=s["sim"])
    return [s["expert"]] if s["sim"] is None else [s["expert"], s["sim"]]


def _prepare_kmeans(case, seed):
    N, K, D = case["N"], case["K"], case["D"]
    rc = mi.planted_router(K, N, D, seed, device=DEV)
    c0 = rc.queries[mi.np_rng(seed, 61).permutation(N)[:K].tolist()].contiguous()   # K of the points, as usual
    return {"x": rc.queries, "router": moin.Router(c0), "assign": torch.empty(N, dtype=torch.int32, device=DEV),
            "plan": moin.Plan(N, K, DEV, moin.PLAN_SEGMENTS), "c_new": torch.empty_like(c0),
            "inv_new": torch.empty(K, dtype=torch.float32, device=DEV)}


def _run_kmeans(case, s):
    moin.route(s["router"], s["x"], out_expert=s["assign"])
    moin.plan_build(s["assign"], case["K"], moin.PLAN_SEGMENTS, plan=s["plan"])
    moin.kmeans_update(s["plan"], s["x"], s["router"].centroids, s["c_new"], s["inv_new"])
    return [s["assign"], s["c_new"], s["inv_new"]]


def _prepare_layer(case, seed):
    E, r, R, K = case["E"], case["r"], case["R"], case["K"]
    lengths = np.asarray(_lengths(case), dtype=np.int64)
    T = int(lengths.sum())
    rng = mi.np_rng(seed, 71)
    rc = mi.planted_router(K, R, case["D"], seed, device=DEV)
    # topics -> experts: the identity where there are as many, else spread; skewed by request for long prompts
    cmap = (np.arange(K) % E).astype(np.int32)
    if E == 5000:
        cmap[rc.labels.cpu().numpy()] = mi.zipf_experts(R, E, 1.1, seed, 72)
    router = moin.Router(rc.centroids, torch.from_numpy(cmap).to(DEV))
    n_slots = max(1, int(round(E * case["kept"])))
    slot = np.full(E, -1, dtype=np.int32)
    slot[np.sort(rng.permutation(E)[:n_slots])] = np.arange(n_slots, dtype=np.int32)
    slot = torch.from_numpy(slot).to(DEV)
    rank = None
    if case["adaptive"]:   # ranks r/8 .. r in multiples of 8
        rank = torch.from_numpy((np.clip((rng.integers(1, 9, n_slots) * r / 8 + 7) // 8 * 8, 8, r)).astype(np.int32)).to(DEV)
    projs = _projections(case)
    xs, ys, jobs = [], [], []
    groups = ((0,),) if case["shape"] == "one" else BLOCK_GROUPS
    for g, group in enumerate(groups):
        x = _normal((T, projs[group[0]][1]), 1.0, seed, 73, g)   # the projections of a group read one input
        xs.append(x)
        row = []
        for p in group:
            _, d_in, d_out = projs[p]
            y = torch.empty(T, d_out, dtype=torch.bfloat16, device=DEV)
            ys.append(y)
            row.append((x, _normal((d_out, d_in), 0.02, seed, 74, p), _pool(E, n_slots, r, d_in, d_out, slot, rank, seed, 75, p), y))
        jobs.append(moin.JobGroup(row))
    # short runs are served by segments (decode), long ones by tiles (prefill), as the decoder chooses
    mode = moin.PLAN_TILES if T // R >= 64 else moin.PLAN_SEGMENTS
    return {"router": router, "queries": rc.queries, "req_expert": torch.empty(R, dtype=torch.int32, device=DEV),
            "token_expert": torch.empty(T, dtype=torch.int32, device=DEV) if T > R else None,
            "request_of_token": torch.from_numpy(np.repeat(np.arange(R), lengths)).to(DEV),
            "plan": moin.Plan(T, E, DEV, mode), "mode": mode, "jobs": jobs, "x": xs, "y": ys,
            "workspace": torch.empty(max(j.workspace_bytes for j in jobs), dtype=torch.uint8, device=DEV)}


def _run_layer(case, s):
    moin.route(s["router"], s["queries"], out_expert=s["req_expert"])
    ids = s["req_expert"]
    if s["token_expert"] is not None:
        ids = torch.index_select(s["req_expert"], 0, s["request_of_token"], out=s["token_expert"])
    moin.plan_build(ids, case["E"], s["mode"], plan=s["plan"])
    for group in s["jobs"]:
        moin.lora_linear_group(s["plan"], group, SCALE, workspace=s["workspace"])
    return [s["req_expert"]] + s["y"]


def _codes(shape, seed, *stream):
    """8-bit float codes of N(0, 1) values and the row scales that make them N(0, 0.02^2) weights."""
    w = _normal(shape, 1.0, seed, *stream)
    return (w.to(torch.float8_e4m3fn).view(torch.uint8).contiguous(),
            torch.full((shape[0],), 0.02, dtype=torch.float32, device=DEV))


def _prepare_forward(case, seed):
    cfg = mi.DecoderConfig(r=case["r"])
    rng = mi.np_rng(seed, 81)
    slot = np.full(cfg.E, -1, dtype=np.int32)
    resident = np.sort(rng.permutation(cfg.E)[:MODEL_SLOTS])
    slot[resident] = np.arange(MODEL_SLOTS, dtype=np.int32)
    slot = torch.from_numpy(slot).to(DEV)
    fp8 = case["base"] == "fp8"
    W, W8, Ws, pools, an, mn = [], [], [], [], [], []
    for l in range(cfg.n_layers):
        an.append(mi.normal_bf16((cfg.hidden,), 0.02, seed, 82, l, device=DEV, mean=1.0))
        mn.append(mi.normal_bf16((cfg.hidden,), 0.02, seed, 83, l, device=DEV, mean=1.0))
        w, w8, ws, pl = {}, {}, {}, {}
        for p, (name, d_in, d_out) in enumerate(cfg.projections()):
            if fp8:
                w8[name], ws[name] = _codes((d_out, d_in), seed, 84, l, p)
            else:
                w[name] = _normal((d_out, d_in), 0.02, seed, 84, l, p)
            pl[name] = _pool(cfg.E, MODEL_SLOTS, cfg.r, d_in, d_out, slot, None, seed, 85, l, p)
        W.append(w); W8.append(w8); Ws.append(ws); pools.append(pl)
    model = moin.DecoderModel(cfg, _normal((cfg.vocab, cfg.hidden), 0.02, seed, 86),
                              _normal((cfg.vocab, cfg.hidden), 0.02, seed, 87),
                              mi.normal_bf16((cfg.hidden,), 0.02, seed, 88, device=DEV, mean=1.0), an, mn, W, pools,
                              cfg.E, SCALE, W8 if fp8 else None, Ws if fp8 else None)
    lengths = _lengths(case)
    b = mi.decoder_batch(cfg, lengths, seed, req_expert=rng.choice(resident, size=case["R"]), device=DEV)
    rows = b.T if case["logits"] == "all" else b.R
    return {"model": model, "tokens": b.tokens, "cu": b.cu_seqlens, "expert": b.req_expert, "max_len": max(lengths),
            "mode": moin.LOGITS_ALL if case["logits"] == "all" else moin.LOGITS_LAST,
            "logits": torch.empty(rows, cfg.vocab, dtype=torch.bfloat16, device=DEV)}


def _run_forward(case, s):
    moin.decoder_forward(s["model"], s["tokens"], s["cu"], s["expert"], s["max_len"], s["mode"], logits=s["logits"])
    return s["logits"]


_PREPARE = {"route": _prepare_route, "kmeans": _prepare_kmeans, "layer": _prepare_layer, "forward": _prepare_forward}
_RUN = {"route": _run_route, "kmeans": _run_kmeans, "layer": _run_layer, "forward": _run_forward}


def prepare(case, seed):
    state = _PREPARE[case["kind"]](case, seed)
    state["case"] = case
    return state


def run(state):
    case = state["case"]
    return _RUN[case["kind"]](case, state)
