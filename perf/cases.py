"""Cases that measure the library through its public entry points: whole prefills, single layers
of a streamed prompt, batches of prompts, layers past the pivot, per-head selection and
block-granular eviction.

Inputs are synthetic and seeded.  A prompt's keys are noise around a set of heavy hitters as large
as the budgets: `kv_budget - window` tokens every later query attends to strongly, and
`struct_budget - kv_budget` more that it attends to less strongly (most of the attention mass sits
on the retained tokens, which is what the method relies on).  The sets that are selected are
therefore separated by a clear gap in the scores and do not hang on the last bit of a sum.
"""
import math

import torch

from paper_2604_06746_b200 import binding, pipeline

DEV = "cuda:0"
HIDDEN = 4096
STRONG, WEAK, SINK = 8.0, 6.0, 9.0      # logit lift of the two sets of heavy hitters and of the first token

# heads, KV heads, head dim
SHAPES = {"llama": (32, 8, 128), "qwen": (28, 4, 128), "small": (8, 2, 64)}


def _case(name, kind, shape, seq, window, budget, layers, dtype="bf16", **more):
    c = {"kind": kind, "shape": shape, "seq": seq, "window": window, "budget": budget, "layers": layers,
         "dtype": dtype, **more}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest whole prefill, fp32 storage: launches and host work
        _case("prefill tiny fp32 2K", "prefill", "small", 2048, 32, 256, 4, "fp32"),
        # an ordinary chat prompt of odd length through all layers of a Llama-shaped model
        _case("prefill llama 5003", "prefill", "llama", 5003, 64, 500, 32),
        # long-document prompts: resident K/V of all layers, 6 to 12 % of it kept
        _case("prefill llama 32K", "prefill", "llama", 32768, 64, 2048, 32),
        _case("prefill llama 128K", "prefill", "llama", 131072, 64, 16384, 32),
        # many query heads per KV head and a window of 128
        _case("prefill qwen 64K", "prefill", "qwen", 65536, 128, 4096, 28),
        # the paper's own default window of 8 queries, on the prompt its overhead is quoted for
        _case("prefill llama 32K window 8", "prefill", "llama", 32768, 8, 3276, 32),
        # a prompt too long to keep all layers: one layer at a time is scored, selected and compacted
        _case("streamed llama 256K", "streamed", "llama", 262144, 64, 8192, 2),
        # the same calls on a short prompt of odd length: latency
        _case("streamed llama 1777", "streamed", "llama", 1777, 64, 177, 4),
        # prompts of different lengths served together
        _case("batch of 4 prompts", "batch", "llama", 131072, 64, 13107, 2, parts="40000,20000,50000,21072"),
        # layers past the pivot: keys gathered at the structural set, scored and selected there
        _case("past the pivot llama 32K", "reduced", "llama", 32768, 64, 2048, 14),
        # every KV head keeps its own tokens
        _case("per-head selection 32K", "heads", "llama", 32768, 64, 3276, 1),
        # block-granular eviction of a paged cache from the accumulated centrality
        _case("paged eviction 128K", "paged", "llama", 131072, 64, 16384, 32, block=16),
    ]


def _size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return n | 1 if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["prefill", "prefill", "prefill", "streamed", "batch", "reduced", "heads", "paged"])
    share = rng.choice([0.05, 0.1, 0.125, 0.2])
    if kind == "prefill":
        shape = rng.choice(["small", "llama", "llama", "qwen"])
        if shape == "small":
            n, dtype = _size(rng, 700, 4096), rng.choice(["fp32", "bf16"])
            return _case(None, kind, shape, n, 32, max(40, int(n * share)), rng.randint(2, 8), dtype)
        window = 128 if shape == "qwen" else rng.choice([8, 16, 32, 64, 64, 64])
        n = _size(rng, 1500, 49152 if shape == "qwen" else 98304)
        return _case(None, kind, shape, n, window, max(window + 8, int(n * share)), rng.randint(8, 28))
    if kind == "streamed":
        n = _size(rng, 1500, 262144)
        return _case(None, kind, "llama", n, 64, max(72, int(n * share)), rng.randint(1, 3))
    if kind == "batch":
        parts = [_size(rng, 1000, 50000) for _ in range(rng.randint(2, 6))]
        n = sum(parts)
        return _case(None, kind, "llama", n, 64, int(n * share), 2, parts=",".join(map(str, parts)))
    if kind == "reduced":
        n = _size(rng, 4000, 65536)
        return _case(None, kind, "llama", n, 64, max(72, int(n * share)), rng.randint(4, 14))
    if kind == "heads":
        n = _size(rng, 2000, 131072)
        return _case(None, kind, "llama", n, 64, max(72, int(n * share)), 1)
    block = rng.choice([16, 32, 64])
    n = block * _size(rng, 100, 131072 // block)
    return _case(None, kind, "llama", n, 64, max(8 * block, int(n * share) // block * block), rng.randint(8, 32),
                 block=block)


# ---- inputs ------------------------------------------------------------------------------------
def _dtype(case):
    return torch.float32 if case["dtype"] == "fp32" else torch.bfloat16


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _struct(case):
    return min(case["seq"], 2 * case["budget"])


def _directions(g, n_kv, d):
    """The direction the window queries of a KV group have in common, of norm sqrt(d)."""
    c = torch.randn((n_kv, d), generator=g, device=DEV)
    return c * (math.sqrt(d) / c.norm(dim=1, keepdim=True))


def _hitters(g, n, window, budget, struct):
    """Positions of the strong and the weak heavy hitters of a prompt (the first token is a strong one)."""
    perm = torch.randperm(n - window - 1, generator=g, device=DEV) + 1
    strong = max(1, budget - window)
    return torch.cat([perm.new_zeros(1), perm[:strong - 1]]), perm[strong - 1:strong - 1 + max(0, struct - budget)]


def _fill_keys(k, c, strong, weak, g):
    """k [H_kv, N, d] in place: noise, 5 % of low-norm delimiters, the heavy hitters along c."""
    d = k.shape[2]
    k.normal_(generator=g)
    k[:, 10::20] *= 0.1
    for pos, lift in ((strong, STRONG), (weak, WEAK)):
        x = torch.randn((k.shape[0], pos.numel(), d), generator=g, device=DEV)
        x += c[:, None] * ((lift - (x @ c[:, :, None]) / math.sqrt(d)) / math.sqrt(d))
        k[:, pos] = x.to(k.dtype)
    k[:, 0] = (k[:, 0].float() + c * ((SINK - STRONG) / math.sqrt(d))).to(k.dtype)


def _queries(g, c, n_heads, window, dtype):
    q = torch.randn((n_heads, window, c.shape[1]), generator=g, device=DEV)
    return (q + c.repeat_interleave(n_heads // c.shape[0], dim=0)[:, None]).to(dtype).contiguous()


def _layers(case, g, strong, weak, with_v=True):
    """Per-layer tensors as a model leaves them.  Attention sharpens at one depth (the pivot)."""
    H, Hkv, d = SHAPES[case["shape"]]
    n, L, dt = case["seq"], case["layers"], _dtype(case)
    turn = int(torch.randint(max(1, L // 4), max(2, 3 * L // 4 + 1), (1,), generator=g, device=DEV))
    jitter = (torch.rand(L, generator=g, device=DEV) * 0.04 + 0.98).tolist()
    out = []
    for l in range(L):
        c = _directions(g, Hkv, d)
        t = {"q_win": _queries(g, c, H, case["window"], dt),
             "scale": 1.0 / (math.sqrt(d) * (1.25 if l < turn else 0.8) * jitter[l])}
        kv = torch.empty((2 if with_v else 1, Hkv, n, d), dtype=dt, device=DEV)
        _fill_keys(kv[0], c, strong, weak, g)
        t["k"] = kv[0]
        if with_v:
            kv[1].normal_(generator=g)
            t["kv"], t["v"] = kv, kv[1]
        out.append(t)
    return out


def _prefill(case, **more):
    H, Hkv, d = SHAPES[case["shape"]]
    return pipeline.Prefill(case["layers"], H, Hkv, d, case["window"], case["seq"], case["budget"], _struct(case),
                            _dtype(case), device=DEV, **more)


def prepare(case, seed):
    g = _gen(seed)
    H, Hkv, d = SHAPES[case["shape"]]
    kind, n, w, B = case["kind"], case["seq"], case["window"], case["budget"]
    s = {"case": case}
    if kind in ("prefill", "streamed", "reduced"):
        strong, weak = _hitters(g, n, w, B, _struct(case))
        s["layers"] = _layers(case, g, strong, weak, with_v=kind != "reduced")
    if kind == "prefill":
        s["pf"] = _prefill(case, hidden_dim=HIDDEN)
        s["hidden"] = torch.randn((n, HIDDEN), generator=g, device=DEV, dtype=torch.bfloat16)
        s["positions"] = torch.arange(n, device=DEV, dtype=torch.int32)
    elif kind == "streamed":
        s["pf"] = _prefill(case, keep_kv=False, defer_head_stats=False)
    elif kind == "reduced":
        s["pf"] = pf = _prefill(case)
        pf.enable_reduced()
        window = torch.arange(n - w, n, device=DEV)
        kept = torch.cat([strong, weak, window]).sort().values.int()
        pf.i_struct.copy_(kept)
        pf.pos_out.copy_(kept)
    elif kind == "batch":
        _prepare_batch(case, g, s)
    else:
        s["ctx"] = binding.Context(H, Hkv, d, w, n, torch.bfloat16, DEV)
        s["kv"] = torch.randn((2, Hkv, n, d), generator=g, device=DEV, dtype=torch.bfloat16)
        if kind == "heads":
            s["cols"] = torch.softmax(2.0 * torch.randn((H, n), generator=g, device=DEV), dim=1)
            s["group"] = torch.empty((Hkv, n), device=DEV)
            s["idx"] = torch.empty((Hkv, B), dtype=torch.int32, device=DEV)
            s["out"] = torch.empty((2, Hkv, B, d), dtype=torch.bfloat16, device=DEV)
        else:
            L, bs = case["layers"], case["block"]
            s["s_hist"] = torch.softmax(1.5 * torch.randn((L, n), generator=g, device=DEV), dim=1) * H
            s["c"] = torch.empty(n, device=DEV)
            s["blocks"] = torch.empty(n // bs, device=DEV)
            s["idx"] = torch.empty(B // bs, dtype=torch.int32, device=DEV)
            s["tokens"] = torch.empty(B, dtype=torch.int32, device=DEV)
            s["recovery"] = torch.empty(L, device=DEV)
            s["out"] = torch.empty((2 * Hkv, B // bs, bs * d), dtype=torch.bfloat16, device=DEV)
    return s


def _prepare_batch(case, g, s):
    H, Hkv, d = SHAPES[case["shape"]]
    n, w, L = case["seq"], case["window"], case["layers"]
    parts = [int(x) for x in case["parts"].split(",")]
    s["cu"] = [sum(parts[:b]) for b in range(len(parts) + 1)]
    s["budgets"] = [max(w + 8, m * case["budget"] // n) for m in parts]
    sets = [_hitters(g, m, w, b, min(m, 2 * b)) for m, b in zip(parts, s["budgets"])]
    s["q"], s["k"] = [], []
    for _ in range(L):
        k = torch.empty((Hkv, n, d), dtype=torch.bfloat16, device=DEV)
        q = torch.empty((len(parts), H, w, d), dtype=torch.bfloat16, device=DEV)
        for b, (strong, weak) in enumerate(sets):
            c = _directions(g, Hkv, d)
            _fill_keys(k[:, s["cu"][b]:s["cu"][b + 1]], c, strong, weak, g)
            q[b] = _queries(g, c, H, w, torch.bfloat16)
        s["q"].append(q)
        s["k"].append(k)
    s["ctx"] = binding.Context(H, Hkv, d, w, max(parts), torch.bfloat16, DEV)
    s["ws"] = s["ctx"].batch_workspace(len(parts), n)
    s["s"] = torch.empty((L, n), device=DEV)
    s["c"] = torch.empty(n, device=DEV)
    s["metrics"] = torch.empty((L, len(parts), 3), device=DEV)
    s["idx"] = torch.empty((L, len(parts), max(s["budgets"])), dtype=torch.int32, device=DEV)


# ---- one pass ------------------------------------------------------------------------------------
def run(s):
    return _RUN[s["case"]["kind"]](s)


def _run_prefill(s):
    """Resident layers: score all, find the pivot, select both budgets, compact K/V and hidden states."""
    pf = s["pf"]
    pivot = pf.run(s["layers"], s["hidden"], s["positions"])
    return {"pivot": pivot, "S": pf.s_hist, "metrics": pf.metrics, "C": pf.c_running, "C*": pf.c_star,
            "I_kv": pf.i_kv, "I_struct": pf.i_struct, "kv": pf.kv_out, "hidden": pf.hidden_out, "pos": pf.pos_out}


def _run_streamed(s):
    """A layer is scored with its metrics, its tokens are selected and compacted, then the next."""
    pf, B = s["pf"], s["case"]["budget"]
    for l, t in enumerate(s["layers"]):
        pf.score(l, t["q_win"], t["k"], t["scale"])
        pf.ctx.select(pf.s_hist[l], B, pf.w, pf.i_kv[l])
        pf.compact_kv(l, t["k"], t["v"], t["kv"])
    return {"S": pf.s_hist, "metrics": pf.metrics, "C": pf.c_running, "I_kv": pf.i_kv, "kv": pf.kv_out}


def _run_batch(s):
    """Packed prompts: every layer scored with metrics for all of them, each prompt's own budget selected."""
    ctx, w, scale = s["ctx"], s["case"]["window"], 1.0 / math.sqrt(s["q"][0].shape[3])
    s["c"].zero_()
    for l in range(len(s["q"])):
        ctx.score_layer_batch(s["q"][l], s["k"][l], s["cu"], scale, s["s"][l], s["metrics"][l], s["ws"], c_inout=s["c"])
        ctx.select_batch(s["s"][l], s["cu"], s["budgets"], w, s["idx"][l])
    return {"S": s["s"], "metrics": s["metrics"], "C": s["c"], "idx": s["idx"]}


def _run_reduced(s):
    """Layers past the pivot, on the keys that survived the truncation."""
    pf = s["pf"]
    for l, t in enumerate(s["layers"]):
        pf.score_reduced(l, t["q_win"], t["k"], t["scale"])
    pf.select_reduced(0, len(s["layers"]))
    return {"S": pf.s_red, "metrics": pf.metrics_red, "I_red": pf.i_red, "I_kv_pos": pf.i_kv_pos, "k": pf.k_red}


def _run_heads(s):
    ctx, case = s["ctx"], s["case"]
    ctx.group_saliency(s["cols"], s["group"])
    ctx.select(s["group"], case["budget"], case["window"], s["idx"])
    ctx.compact_per_slab(s["kv"][0], s["idx"], s["out"][0])
    ctx.compact_per_slab(s["kv"][1], s["idx"], s["out"][1])
    return {"group": s["group"], "idx": s["idx"], "kv": s["out"]}


def _run_paged(s):
    """Centrality at the pivot, pooled per block, best blocks kept and gathered, share of the attention kept."""
    ctx, case = s["ctx"], s["case"]
    bs, kv = case["block"], s["kv"]
    ctx.accumulate(s["s_hist"], case["layers"] // 2, 0.9, s["c"])
    ctx.block_scores(s["c"], bs, s["blocks"])
    ctx.select(s["blocks"], s["idx"].numel(), max(1, case["window"] // bs), s["idx"])
    ctx.compact(kv.view(2 * kv.shape[1], -1, bs * kv.shape[3]), s["idx"], s["out"])
    ctx.select(s["c"], s["tokens"].numel(), case["window"], s["tokens"])
    ctx.mass_recovery(s["s_hist"], s["tokens"], s["recovery"])
    return {"c": s["c"], "blocks": s["blocks"], "idx": s["idx"], "tokens": s["tokens"], "kv": s["out"],
            "recovery": s["recovery"]}


_RUN = {"prefill": _run_prefill, "streamed": _run_streamed, "batch": _run_batch, "reduced": _run_reduced,
        "heads": _run_heads, "paged": _run_paged}


# ---- what a pass cannot do without -----------------------------------------------------------------
def work(case):
    H, Hkv, d = SHAPES[case["shape"]]
    n, w, B, L, kind = case["seq"], case["window"], case["budget"], case["layers"], case["kind"]
    e = 4 if case["dtype"] == "fp32" else 2
    keys, row = Hkv * n * d * e, Hkv * d * e
    flops = 2 * H * w * n * d
    if kind == "prefill":       # K once, the kept V rows in, K and V rows out, S, index lists; hidden rows and C
        hidden = _struct(case) * (2 * HIDDEN * 2 + 3 * 4)
        return {"bytes": L * (keys + H * w * d * e + 3 * B * row + 4 * n + 4 * B) + hidden + 8 * n, "flops": L * flops}
    if kind == "streamed":
        return {"bytes": L * (keys + H * w * d * e + 3 * B * row + 4 * n + 4 * B) + 4 * n, "flops": L * flops}
    if kind == "batch":
        P = case["parts"].count(",") + 1
        return {"bytes": L * (keys + P * H * w * d * e + 4 * n + 4 * B) + 4 * n, "flops": L * flops}
    if kind == "reduced":       # the kept K rows in (out once, for the layer that stays), S and index lists
        m = _struct(case)
        return {"bytes": L * (m * row + H * w * d * e + 4 * m + 8 * B) + m * row, "flops": L * 2 * H * w * m * d}
    if kind == "heads":
        return {"bytes": 4 * H * n + 4 * Hkv * n + 4 * Hkv * B + 4 * B * row, "flops": H * n}
    return {"bytes": 4 * L * n + 4 * n + 4 * n // case["block"] + 4 * B * row + 4 * B, "flops": 2 * L * n}


def tolerance(case):
    if case["kind"] == "heads":
        return "exact"
    if case["kind"] == "paged" or case["dtype"] == "fp32":
        return {"rel": 1e-5}
    # bf16 storage: exact products in fp32 accumulators, exponentials good to 1e-4 and sums of thousands of them
    return {"rel": 1e-4}
