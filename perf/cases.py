"""Workloads whose speed is tracked, each driven through the public entry points of the library.

A case is a dict of plain values.  `kind` says what the caller does with the library:

  decode    one image batch: every layer at every scale through hack_scale_step
  staged    the same loop through hack_score, hack_select, hack_compact, hack_attend
  host      the same loop from pinned host buffers (hack_scale_step_host)
  classify  offline head classification: an uncompressed cache is decoded up to the last scale, whose
            attention also returns the variance of every head (hack_attend_variance)
  score     importance scores of dense tensors without a cache (hack_score_noalloc)

A decode pass walks the scales in order and all layers inside a scale, as the model does, on inputs
that are resident before the pass; the inputs and outputs of the stack are far larger than the L2
cache except in the smallest cases.
"""
import math

import torch

import paper_2504_09261_b200 as hb

SIDES_256 = "1,2,3,4,5,6,8,10,13,16"                  # 680 tokens
SIDES_512 = "1,2,3,4,6,9,13,18,24,32"                 # 2240 tokens
SIDES_1024 = "1,2,4,6,8,12,16,20,24,32,40,48,64"      # 10521 tokens


def _loop(name, kind, dtype, layers, heads, dim, batch, sides, alpha, budget_c, budget_s, n_obs=32, compete=False, merge=False):
    return {"name": name, "kind": kind, "dtype": dtype, "layers": layers, "heads": heads, "dim": dim, "batch": batch,
            "sides": sides, "alpha": alpha, "budget_c": budget_c, "budget_s": budget_s, "n_obs": n_obs,
            "compete": compete, "merge": merge}


def listed():
    return [
        # one fp32 layer, one image of 256 x 256: the exact-precision path at its smallest, all latency
        _loop("f32-256-one-layer", "decode", "f32", 1, 16, 64, 1, SIDES_256, 0.5, 34, 374),
        # fp32 at 512 x 512 through the stage calls: what a study of the method's parts runs
        _loop("f32-512-staged", "staged", "f32", 2, 16, 128, 1, SIDES_512, 0.4, 224, 1717, n_obs=16),
        # one 256 x 256 image through a 16-layer stack: the latency a single request sees
        _loop("d16-256-bs1", "decode", "bf16", 16, 16, 64, 1, SIDES_256, 0.5, 68, 612),
        # the same stack serving a batch of 16
        _loop("d16-256-bs16", "decode", "bf16", 16, 16, 64, 16, SIDES_256, 0.5, 68, 612),
        # 512 x 512, 30 layers of 30 heads, batch 8, budget 30 %
        _loop("d30-512-bs8", "decode", "bf16", 30, 30, 64, 8, SIDES_512, 0.4, 112, 1045),
        # 1024 x 1024, 32 layers of 16 heads, conditional and unconditional branch, budget 30 %: the headline
        _loop("2b-1024-bs2", "decode", "bf16", 32, 16, 128, 2, SIDES_1024, 0.5, 2104, 4208),
        # 1024 x 1024, 40 layers of 32 heads: the largest
        _loop("8b-1024-bs2", "decode", "bf16", 40, 32, 128, 2, SIDES_1024, 0.5, 2104, 4208),
        # odd sides, odd head count and batch, the current scale competes for the budget, 24 observation rows
        _loop("ragged-compete", "decode", "bf16", 6, 7, 128, 3, "1,3,5,7,9,11,15,19,27,37,45", 0.6, 475, 951, n_obs=24,
              compete=True),
        # the last scale folds what contextual heads discard into what they keep
        _loop("2b-1024-merge", "decode", "bf16", 4, 16, 128, 2, SIDES_1024, 0.5, 2104, 4208, merge=True),
        # four layers of a head-classification sample: uncompressed cache, variance at the last scale
        _loop("classify-1024", "classify", "bf16", 4, 16, 128, 2, SIDES_1024, 0.5, 10521, 10521),
        # Q, K and V arrive in pinned host memory and the result goes back there
        _loop("host-256-bs8", "host", "bf16", 4, 16, 64, 8, SIDES_256, 0.5, 68, 612),
        # scores for a server that may not allocate: 32 heads against 2000 candidate keys
        {"name": "score-dense", "kind": "score", "dtype": "bf16", "rows": 32, "queries": 1024, "cand": 2000, "dim": 128, "n_obs": 32},
    ]


# ------------------------------------------------------------------ drawn cases
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode"] * 8 + ["staged", "host", "classify", "score"])
    if kind == "score":
        rows = _log_int(rng, 4, 512)
        return {"kind": kind, "dtype": rng.choice(["bf16", "f32"]), "rows": rows, "queries": _log_int(rng, 16, 4096),
                "cand": _log_int(rng, 64, 65536 // rows), "dim": rng.choice([64, 128]), "n_obs": rng.choice([8, 16, 32, 32])}
    dtype = "f32" if kind in ("decode", "staged") and rng.random() < 0.2 else "bf16"
    # a schedule that grows from 1 to its last side, with odd sides on the way
    last, n = _log_int(rng, 10, 32 if dtype == "f32" or kind == "host" else 64), rng.randint(8, 13)
    sides = [1]
    for i in range(1, n):
        side = int(round(last ** (i / (n - 1)) * rng.uniform(0.85, 1.15)))
        if side > sides[-1]:
            sides.append(side)
    tokens = sum(s * s for s in sides)
    alpha = round(rng.uniform(0.25, 0.75), 2)
    budget_c = max(8, int(rng.uniform(0.1, 0.6) * tokens / (alpha + 2 * (1 - alpha))))
    case = {"kind": kind, "dtype": dtype, "layers": 1, "heads": rng.randint(6, 32), "dim": rng.choice([64, 128]),
            "batch": _log_int(rng, 1, 4 if dtype == "f32" else 16), "sides": ",".join(str(s) for s in sides), "alpha": alpha,
            "budget_c": budget_c, "budget_s": min(2 * budget_c, tokens), "n_obs": rng.choice([8, 16, 32, 32, 32]),
            "compete": rng.random() < 0.25, "merge": kind == "decode" and dtype == "bf16" and rng.random() < 0.1}
    if kind == "classify":
        case.update(budget_c=tokens, budget_s=tokens, compete=False)
    # as many layers, up to a whole stack, as stay well below the largest listed case
    one = work(case)
    most = {"host": 0.2e9, "classify": 3e9}.get(kind, 10e9) / one["bytes"]
    most = min(most, (0.1e12 if dtype == "f32" else 12e12) / one["flops"])
    case["layers"] = max(1, min(_log_int(rng, 1, 40), int(most)))
    while case["batch"] > 1 and work(case)["bytes"] > 12e9:
        case["batch"] //= 2
    return case


# ------------------------------------------------------------------ one pass
def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def _sides(case):
    return [int(s) for s in case["sides"].split(",")]


def _position_code(side, side_max, dim, device):
    """2-D sinusoidal code of a scale's token grid, squared norm sqrt(dim)."""
    c = (torch.arange(side, device=device, dtype=torch.float32) + 0.5) / side
    omega = 2 * math.pi * (side_max / 2.0) ** torch.linspace(0, 1, dim // 4, device=device)
    y = (c.view(side, 1, 1) * omega).expand(side, side, dim // 4)
    x = (c.view(1, side, 1) * omega).expand(side, side, dim // 4)
    code = torch.cat([y.sin(), y.cos(), x.sin(), x.cos()], dim=-1).reshape(side * side, dim)
    return code * math.sqrt(math.sqrt(dim) / (dim / 2.0))


def _inputs(case, seed, device):
    """Head mask and per scale Q, K, V [layers, batch, heads, N_k, dim] with the two attention patterns of
    visual autoregressive stacks: contextual heads attend to a few sink keys, structural heads to the
    neighbourhood of the query's position; values are N(0, 1)."""
    L, H, b, D, sides = case["layers"], case["heads"], case["batch"], case["dim"], _sides(case)
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    n_ctx = min(max(int(round(case["alpha"] * L * H)), 1), L * H)
    order = torch.randperm(L * H, generator=torch.Generator().manual_seed(seed))
    mask = torch.zeros(L * H, dtype=torch.uint8)
    mask[order[:n_ctx]] = 1
    mask = mask.view(L, H)
    ctx = mask.to(device).float().view(L, 1, H, 1, 1)
    u = torch.randn((L, 1, H, 1, D), generator=gen, device=device)
    u = 4.0 * u / u.norm(dim=-1, keepdim=True) * ctx
    qkv = []
    for side in sides:
        shape = (L, b, H, side * side, D)
        p = 3.0 * _position_code(side, sides[-1], D, device) * (1.0 - ctx)
        sink = (torch.rand((L, 1, H, side * side, 1), generator=gen, device=device) < 0.01).float()
        q = torch.randn(shape, generator=gen, device=device).add_(u).add_(p).to(_dtype(case))
        k = torch.randn(shape, generator=gen, device=device).add_(u * sink).add_(p).to(_dtype(case))
        v = torch.randn(shape, generator=gen, device=device).to(_dtype(case))
        qkv.append((q, k, v))
    return mask, qkv


def prepare(case, seed):
    device = torch.device("cuda:0")
    if case["kind"] == "score":
        gen = torch.Generator(device=device)
        gen.manual_seed(seed)
        rows, D = case["rows"], case["dim"]
        q = torch.randn((rows, case["queries"], D), generator=gen, device=device).to(_dtype(case))
        k = torch.randn((rows, case["cand"], D), generator=gen, device=device).to(_dtype(case))
        return {"case": case, "q": q, "k": k, "scores": torch.empty((rows, case["cand"]), device=device)}
    mask, qkv = _inputs(case, seed, device)
    cache = hb.HackCache(case["layers"], case["heads"], case["dim"], case["batch"], _sides(case),
                         hb.HACK_F32 if case["dtype"] == "f32" else hb.HACK_BF16, mask, case["budget_c"],
                         case["budget_s"], n_obs=case["n_obs"], overflow_policy=int(case["compete"]), device=0,
                         merge_last=case["merge"])
    outs = [torch.empty_like(q) for q, _, _ in qkv]
    if case["kind"] == "host":
        qkv = [tuple(t.cpu().pin_memory() for t in s) for s in qkv]
        outs = [t.cpu().pin_memory() for t in outs]
    bh = case["batch"] * case["heads"]
    state = {"case": case, "cache": cache, "outs": outs,
             # per scale and layer: q, k, v, out
             "steps": [[(q[l], k[l], v[l], o[l]) for l in range(case["layers"])] for (q, k, v), o in zip(qkv, outs)]}
    if case["kind"] in ("staged", "classify"):
        state["scores"] = torch.empty((bh, cache.cand_stride), device=device)
        state["idx"] = torch.empty((bh, cache.kept_stride), dtype=torch.int32, device=device)
    if case["kind"] == "classify":
        state["sigma"] = torch.zeros((case["layers"], bh), device=device)
    return state


def run(state):
    case = state["case"]
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "score":
        hb.hack_score_noalloc(state["q"], state["k"], state["scores"], case["rows"], case["queries"], case["cand"],
                              case["cand"], case["dim"], hb.HACK_F32 if case["dtype"] == "f32" else hb.HACK_BF16,
                              case["n_obs"], 0.0, stream)
        return state["scores"]
    cache, steps = state["cache"], state["steps"]
    cache.hack_reset()
    if case["kind"] == "decode":
        for k, scale in enumerate(steps):
            for l, (q, kk, v, out) in enumerate(scale):
                cache.hack_scale_step(l, k, q, kk, v, out, stream)
        return state["outs"]
    if case["kind"] == "host":
        for k, scale in enumerate(steps):
            for l, (q, kk, v, out) in enumerate(scale):
                cache.hack_scale_step_host(l, k, q, kk, v, out, stream)
        return state["outs"]
    scores, idx = state["scores"], state["idx"]
    variance_at = len(steps) - 1 if case["kind"] == "classify" else -1
    for k, scale in enumerate(steps):
        for l, (q, kk, v, out) in enumerate(scale):
            if case["kind"] == "classify" and k != variance_at:
                cache.hack_scale_step(l, k, q, kk, v, out, stream)
                continue
            cache.hack_score(l, k, q, kk, scores, stream)
            cache.hack_select(l, k, scores, idx, None, stream)
            cache.hack_compact(l, k, idx, kk, v, stream)
            if k == variance_at:
                cache.hack_attend_variance(l, k, q, out, state["sigma"][l], stream)
            else:
                cache.hack_attend(l, k, q, out, stream)
    return state["outs"] + ([state["sigma"]] if case["kind"] == "classify" else [])


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Q, K, V read and O written once per step; of the cache, the stored keys of a head and the stored
    values it keeps are read once per step and the rows by which the cache grows are written.  Scoring
    reads every candidate key (already counted) and costs 2 n_obs D per key of a head over its budget;
    attention 4 N_k D per key kept, and the variance pass forms Q K^T once more."""
    e, D = (4 if case["dtype"] == "f32" else 2), case["dim"]
    if case["kind"] == "score":
        n_obs = min(case["n_obs"], case["queries"])
        return {"bytes": case["rows"] * (case["cand"] * (D * e + 4) + n_obs * D * e),
                "flops": 2.0 * case["rows"] * case["cand"] * n_obs * D}
    units = case["layers"] * case["heads"]
    n_ctx = min(max(int(round(case["alpha"] * units)), 1), units)
    sides = _sides(case)
    t_init = sum(s * s for s in sides[:2])
    rows = flops = 0.0
    for contextual, heads in ((True, n_ctx * case["batch"]), (False, (units - n_ctx) * case["batch"])):
        budget, stored = (case["budget_c"] if contextual else case["budget_s"]), 0
        for k, side in enumerate(sides):
            n, cand = side * side, stored + side * side
            kept = cand
            if cand > budget:
                protected = min(stored, t_init) + (0 if case["compete"] else n)
                kept = budget if contextual else cand if k < 2 else min(cand, max(budget, protected))
                flops += heads * 2.0 * min(case["n_obs"], n) * D * cand
            flops += heads * (6.0 if case["kind"] == "classify" and k == len(sides) - 1 else 4.0) * n * D * kept
            rows += heads * (4 * n + stored + min(stored, kept) + 2 * max(kept - stored, 0))
            stored = kept
    return {"bytes": rows * D * e, "flops": flops}


def tolerance(case):
    """bf16 outputs carry one rounding of the result and one of the probabilities (2.3e-3 against 64-bit
    attention over the same rows); fp32 results differ by the order of their sums (outputs 1.2e-6 at 2240
    keys, scores 1.4e-7).  A selection decided the other way at a near-tie swaps one barely attended key of
    one head."""
    if case["kind"] == "score":
        return {"rel": 1e-6}
    return {"rel": 1e-5 if case["dtype"] == "f32" else 1e-2}
