"""The work that users of the AudioKV eviction pass have it do, as cases that can be timed and compared.

A case names an entry point (`api`) and the shape it meets. K, V, Q and the head scores follow the recipe of
`paper_2604_06694_b200.workloads`: audio rows are an AR(1) process along the tokens, text rows are independent, the
leading tokens may be attention sinks; they are drawn on the GPU here because they are drawn often. Heads differ in how
sharply they attend: the queries of a KV head's group carry a gain drawn from [sharp_lo, sharp_hi]. With logits of
standard deviation 2 a head's scores are nearly flat and its spectrum is mostly mean; from about 3 on a few tokens hold
most of the attention and the energy spreads over the whole spectrum. Models have heads of both kinds.
"""
import math

import numpy as np
import torch

from paper_2604_06694_b200 import binding as B


def _case(name, api, dtype, layers, hq, hkv, d, lens, **more):
    c = {"name": name, "api": api, "dtype": dtype, "layers": layers, "hq": hq, "hkv": hkv, "d": d, "lens": lens,
         "window": 32, "keep": 0.4, "sinks": 0, "sharp_lo": 1.5, "sharp_hi": 3.5, "page": 0, "mode": 0}
    c.update(more)
    return c


def listed():
    return [
        # The smallest call: one fp32 layer of a short prompt, as a unit of a test or a notebook. Latency is all of it.
        _case("one_layer_f32_1k", "evict", "f32", 1, 8, 2, 64, "1024", sinks=1),
        # A server that answers short voice turns: the prompts have lengths of their own, one context serves them all,
        # and each is evicted when its prefill ends. Every call brings a shape that the call before it did not have.
        _case("voice_turns_7b", "turns", "bf16", 28, 28, 4, 128, "655,412,1571,1038"),
        # The benchmark's shape: one 8k prompt of the 7B stack.
        _case("prompt_7b_8k", "evict", "bf16", 28, 28, 4, 128, "8192", sharp_hi=2.5),
        # Long audio, the same stack.
        _case("prompt_7b_32k", "evict", "bf16", 28, 28, 4, 128, "32768"),
        # The deepest stack, with attention sinks.
        _case("prompt_30b_16k_sinks", "evict", "bf16", 48, 32, 4, 128, "16384", sinks=4),
        # A ragged batch of eight requests at head_dim 256 in one call.
        _case("batch8_e4b_ragged", "evict", "bf16", 35, 8, 2, 256, "2573,19873,4110,31415,7001,2999,11213,6955"),
        # A serving stack's block allocator: token-major pages of 16 tokens, four requests, a smaller cache kept.
        _case("paged_batch4_7b", "evict", "bf16", 28, 28, 4, 128, "1181,2750,4093,6400", page=16, keep=0.25),
        # The decode direction: a compacted cache, ragged per head, that has grown by 128 tokens and is cut back.
        _case("reevict_7b", "reevict", "bf16", 28, 28, 4, 128, "8192", new=128),
        # The 7B stack held in fp32, as for an accuracy study.
        _case("prompt_f32_4k", "evict", "f32", 28, 28, 4, 128, "4096"),
        # The steps called one by one on an odd length, with the cut-off that leaves the mean out, and the spread
        # statistic of what was kept: an ablation run.
        _case("steps_7b_12k_odd", "steps", "bf16", 28, 28, 4, 128, "12001", mode=B.AUDIOKV_SMOOTH_ENERGY_NO_MEAN,
              window=16),
        # The offline head score: recorded attention rows of 64 decode steps, 784 heads.
        {"name": "hit_score_8k", "api": "hit", "steps": 64, "heads": 784, "audio": 8112, "top_k": 24},
        # The cache in pinned host memory, the whole call: copies in, pass, copies out.
        _case("host_7b_8k", "host", "bf16", 28, 28, 4, 128, "8192", sharp_hi=2.5),
    ]


#: (query heads, KV heads, head_dim, layers) of the stacks above
_STACKS = [(28, 4, 128, 28), (32, 4, 128, 48), (8, 2, 256, 35), (8, 2, 64, 16)]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    api = rng.choice(["evict", "evict", "evict", "ragged", "paged", "f32", "turns", "reevict", "steps", "hit", "host"])
    if api == "hit":
        return {"api": "hit", "steps": rng.randint(4, 64), "heads": _log_int(rng, 32, 784),
                "audio": _log_int(rng, 700, 8112), "top_k": rng.choice([8, 24, 24, 64])}
    hq, hkv, d, layers = rng.choice(_STACKS)
    layers = max(1, layers - rng.choice([0, 0, layers // 4, layers // 2]))
    more = {"window": rng.choice([16, 32, 32, 64] if hq // hkv * 64 <= 512 else [16, 32]),
            "keep": round(rng.uniform(0.2, 0.6), 3), "sinks": rng.choice([0, 0, 1, 4]),
            "sharp_lo": 1.5, "sharp_hi": rng.choice([2.5, 3.5, 3.5])}
    dtype = "bf16"
    if api == "ragged":
        lens = [_log_int(rng, 700, 12000) for _ in range(rng.randint(2, 8))]
        api = "evict"
    elif api == "paged":
        lens = [_log_int(rng, 700, 8000) for _ in range(rng.randint(1, 4))]
        more["page"] = rng.choice([16, 16, 32, 64, 128])
        api = "evict"
    elif api == "turns":
        lens = [_log_int(rng, 350, 3000) for _ in range(rng.randint(2, 6))]
    elif api == "f32":
        lens = [_log_int(rng, 700, 4096)]
        dtype, api = "f32", "evict"
    elif api == "reevict":
        lens = [_log_int(rng, 1500, 12000) for _ in range(rng.choice([1, 1, 2]))]
        more["new"] = rng.choice([32, 64, 128, 256])
        more["window"] = min(more["window"], more["new"])
    elif api == "steps":
        lens = [_log_int(rng, 700, 12001)]
        more["mode"] = rng.choice([B.AUDIOKV_SMOOTH_SSS, B.AUDIOKV_SMOOTH_ENERGY_NO_MEAN, B.AUDIOKV_SMOOTH_AVG_POOL])
    elif api == "host":
        lens = [_log_int(rng, 700, 8192)]
        layers = max(2, layers // 2)
    else:
        lens = [_log_int(rng, 700, 32768)]
    c = _case("", api, dtype, layers, hq, hkv, d, ",".join(str(x) for x in lens), **more)
    del c["name"]
    return c


def _lens(c):
    return [int(x) for x in c["lens"].split(",")]


def _torch_dtype(c):
    return torch.float32 if c["dtype"] == "f32" else torch.bfloat16


def _ar1_(x, rho):
    """x[h, t] <- rho_h x[h, t-1] + sqrt(1 - rho_h^2) x[h, t] along dim 1, in place, by doubling strides."""
    x *= torch.sqrt(1 - rho * rho)
    x[:, 0] /= torch.sqrt(1 - rho[:, 0] * rho[:, 0])
    s, p = 1, rho.clone()
    while s < x.shape[1] and s < 2048:  # 0.99^2048 is below fp32 rounding
        x[:, s:] += p * x[:, :-s].clone()
        p = p * p
        s *= 2


def _rows(gen, heads, n, n_audio, d, rho):
    x = torch.randn((heads, n, d), generator=gen, device="cuda")
    if n_audio > 1:
        _ar1_(x[:, :n_audio], rho)
    return x


def _uniform(gen, n, lo, hi):
    return lo + (hi - lo) * torch.rand((n, 1, 1), generator=gen, device="cuda")


def _queries(c, gen, n_req):
    W, hkv, G, d = c["window"], c["hkv"], c["hq"] // c["hkv"], c["d"]
    q = torch.randn((n_req, c["layers"], W, hkv, G, d), generator=gen, device="cuda")
    gain = c["sharp_lo"] + (c["sharp_hi"] - c["sharp_lo"]) * torch.rand((1, c["layers"], 1, hkv, 1, 1), generator=gen,
                                                                        device="cuda")
    return (q * gain).to(_torch_dtype(c)).reshape(n_req, c["layers"], W, c["hq"], d)


def _q_strides(c):
    tok = c["hq"] * c["d"]
    return (c["layers"] * c["window"] * tok, c["window"] * tok, tok, c["d"])


def _caches(c, gen):
    """K and V of the case's requests, [layer][head][token][d] (requests one after another along the tokens)."""
    lens, d = _lens(c), c["d"]
    k, v = (torch.empty((c["layers"], c["hkv"], sum(lens), d), dtype=_torch_dtype(c), device="cuda") for _ in range(2))
    at = 0
    for L in lens:
        n_audio = int(0.9 * L)
        for layer in range(c["layers"]):
            rho = _uniform(gen, c["hkv"], 0.85, 0.99)
            x = _rows(gen, c["hkv"], L, n_audio, d, rho)
            if c["sinks"]:
                x[:, :c["sinks"]] *= 8.0
            k[layer, :, at:at + L] = x
            v[layer, :, at:at + L] = _rows(gen, c["hkv"], L, n_audio, d, rho)
        at += L
    return k, v


def _paged(c, gen, k, v):
    """The same caches in pools of pages handed out in a random order: [layer][pool row][head][d], and the table."""
    lens, ps = _lens(c), c["page"]
    per = [-(-L // ps) for L in lens]
    n_pages = sum(per) + 3
    order = torch.randperm(n_pages, generator=gen, device="cuda")[:sum(per)]
    table = torch.full((len(lens), max(per)), -1, dtype=torch.int32, device="cuda")
    rows, at = [], 0
    for r, L in enumerate(lens):
        pages = order[at:at + per[r]]
        table[r, :per[r]] = pages.to(torch.int32)
        rows.append((pages[:, None] * ps + torch.arange(ps, device="cuda")).reshape(-1)[:L])
        at += per[r]
    rows = torch.cat(rows)
    pools = []
    for t in (k, v):
        pool = torch.zeros((c["layers"], n_pages * ps, c["hkv"], c["d"]), dtype=t.dtype, device="cuda")
        pool[:, rows] = t.transpose(1, 2)
        pools.append(pool)
    return pools[0], pools[1], table, n_pages


def _problem(c, lens, kv_strides, kv_req_offset=None, **more):
    base = max(0, int(0.1 * (math.floor(c["keep"] * min(lens)) - c["window"])))
    return B.Problem(B.AUDIOKV_F32 if c["dtype"] == "f32" else B.AUDIOKV_BF16, c["layers"], c["hq"], c["hkv"], c["d"],
                     lens, c["window"], _q_strides(c), kv_strides, kv_req_offset=kv_req_offset, base_per_head=base,
                     smooth_mode=c["mode"], pool_kernel=7 if c["mode"] >= B.AUDIOKV_SMOOTH_AVG_POOL else 1, **more)


def _budgets(c, lens):
    n = c["layers"] * c["hkv"]
    return [B.audiokv_budget_from_ratio(c["keep"], n, L, c["window"]) for L in lens]


def _head_scores(c, seed, n_req):
    s = np.random.default_rng(seed).beta(0.5, 2.0, size=(n_req, c["layers"], c["hkv"]))
    return torch.from_numpy(s.astype(np.float32)).cuda()


def _outputs(c, rows, heads, device="cuda"):
    pin = device == "cpu"
    o = {n: torch.zeros((rows, c["d"]), dtype=_torch_dtype(c), device=device, pin_memory=pin) for n in ("k_out", "v_out")}
    o["kept_idx"] = torch.zeros(rows, dtype=torch.int32, device=device, pin_memory=pin)
    o["budgets"] = torch.zeros(heads, dtype=torch.int32, device=device, pin_memory=pin)
    o["cu_kept"] = torch.zeros(heads + 1, dtype=torch.int32, device=device, pin_memory=pin)
    return o


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return {"evict": _prepare_evict, "turns": _prepare_turns, "reevict": _prepare_reevict, "steps": _prepare_steps,
            "hit": _prepare_hit, "host": _prepare_host}[c["api"]](c, gen, int(seed))


def _prepare_evict(c, gen, seed):
    lens = _lens(c)
    k, v = _caches(c, gen)
    if c["page"]:
        k, v, table, n_pages = _paged(c, gen, k, v)
        strides = (n_pages * c["page"] * c["hkv"] * c["d"], c["hkv"] * c["d"], c["d"])
        prob = _problem(c, lens, strides, page_size=c["page"], n_pages=n_pages, page_table=table)
    else:
        starts = np.concatenate([[0], np.cumsum(lens)[:-1]])
        strides = (c["hkv"] * sum(lens) * c["d"], c["d"], sum(lens) * c["d"])
        prob = _problem(c, lens, strides, [int(s) * c["d"] for s in starts])
    budgets = _budgets(c, lens)
    return {"c": c, "prob": prob, "ctx": B.Context(prob), "q": _queries(c, gen, len(lens)), "k": k, "v": v,
            "S": _head_scores(c, seed, len(lens)), "budget": budgets, "out": _outputs(c, sum(budgets), prob.total_heads)}


def _turn_problem(c, L):
    return _problem(c, [L], (c["hkv"] * L * c["d"], c["d"], L * c["d"]))


def _prepare_turns(c, gen, seed):
    turns = []
    for i, L in enumerate(_lens(c)):
        one = dict(c, lens=str(L))
        k, v = _caches(one, gen)
        budget = _budgets(c, [L])
        turns.append({"L": L, "q": _queries(c, gen, 1), "k": k, "v": v, "S": _head_scores(c, seed + 7919 * i, 1),
                      "budget": budget, "out": _outputs(c, sum(budget), c["layers"] * c["hkv"])})
    probs = [_turn_problem(c, t["L"]) for t in turns]
    size = max(B.audiokv_workspace_bytes(p) for p in probs)
    return {"c": c, "turns": turns, "ctx": B.Context(probs[0], workspace_bytes=size)}


def _prepare_reevict(c, gen, seed):
    W, d = c["window"], c["d"]
    rng = np.random.default_rng(seed)
    heads, keep = c["layers"] * c["hkv"], []
    for L in _lens(c):  # budgets spread evenly from half to one and a half times the mean, dealt out over the heads
        share = 0.5 + (rng.permutation(heads) + 0.5) / heads
        keep += [min(L, max(W + 1, int(round(c["keep"] * L * x)))) for x in share]
    cu = [0]
    for b in keep:
        cu.append(cu[-1] + b + c["new"])
    k, v = (torch.empty((cu[-1], d), dtype=_torch_dtype(c), device="cuda") for _ in range(2))
    for u, b in enumerate(keep):
        rho = _uniform(gen, 1, 0.85, 0.99)
        x = _rows(gen, 1, b + c["new"], b, d, rho)[0]
        if c["sinks"]:
            x[:c["sinks"]] *= 8.0
        k[cu[u]:cu[u + 1]] = x
        v[cu[u]:cu[u + 1]] = _rows(gen, 1, b + c["new"], b, d, rho)[0]
    prob = _problem(c, _lens(c), (0, d, 0))
    ctx = B.Context(prob, workspace_bytes=B.audiokv_reevict_workspace_bytes(prob, cu))
    return {"c": c, "prob": prob, "ctx": ctx, "q": _queries(c, gen, len(_lens(c))), "k": k, "v": v, "cu": cu,
            "keep": keep, "out": _outputs(c, sum(keep), len(keep))}


def _prepare_steps(c, gen, seed):
    s = _prepare_evict(c, gen, seed)
    n = B.audiokv_scores_len(s["prob"])
    s["scores"] = torch.zeros(n, device="cuda")
    s["smoothed"] = torch.zeros(n, device="cuda")
    s["kstar"] = torch.zeros(s["prob"].total_heads, dtype=torch.int32, device="cuda")
    s["hist"] = torch.zeros((len(_lens(c)), 64), dtype=torch.int32, device="cuda")
    s["stats"] = torch.zeros((len(_lens(c)), 2), device="cuda")
    return s


def _hit_lens(c):
    return [c["audio"] + 16 + t for t in range(c["steps"])]


def _prepare_hit(c, gen, seed):
    T, H, width = c["steps"], c["heads"], c["audio"] + 16 + c["steps"]
    attn = torch.zeros((T, H, width), device="cuda")
    ground = torch.from_numpy(np.random.default_rng(seed).beta(0.5, 2.0, size=(H, 1)).astype(np.float32)).cuda()
    spans = []
    for t, L in enumerate(_hit_lens(c)):
        lo = min(c["audio"] - 12, int(t * (c["audio"] - 12) / max(1, T - 1)))
        spans.append((lo, lo + 11))
        z = torch.randn((H, L), generator=gen, device="cuda")
        z[:, 0] += 4.0
        z[:, lo:lo + 12] += 6.0 * ground
        attn[t, :, :L] = torch.softmax(z, dim=1)
    prob = B.Problem(B.AUDIOKV_F32, 1, 1, 1, 64, [64], 1, (64, 64, 64, 64), (64 * 64, 64, 64 * 64))
    return {"c": c, "ctx": B.Context(prob), "attn": attn,
            "row_len": torch.tensor(_hit_lens(c), dtype=torch.int32, device="cuda"),
            "span": torch.tensor(spans, dtype=torch.int32, device="cuda"),
            "counts": torch.zeros(H, dtype=torch.int32, device="cuda"), "s_hit": torch.zeros(H, device="cuda")}


def _prepare_host(c, gen, seed):
    s = _prepare_evict(c, gen, seed)
    for n in ("q", "k", "v", "S"):
        t = s.pop(n)
        s[n] = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
        s[n].copy_(t)
    s["out"] = _outputs(c, sum(s["budget"]), s["prob"].total_heads, "cpu")
    size = B.audiokv_workspace_bytes_host(s["prob"], s["q"].numel(), s["k"].numel(), s["budget"])
    s["ctx"] = B.Context(s["prob"], workspace_bytes=size)
    return s


def _bits(o):
    """The outputs; K and V rows are copies of input bits, so they are handed over as whole numbers."""
    return {n: t.view(torch.int16 if t.dtype == torch.bfloat16 else torch.int32) for n, t in o.items()}


def _evict(ctx, prob, s, call=B.audiokv_evict):
    o = s["out"]
    call(ctx, prob, s["q"], s["k"], s["v"], s["S"], s["budget"], o["k_out"], o["v_out"], o["kept_idx"], o["budgets"],
         o["cu_kept"])
    return _bits(o)


def run(state):
    s, api = state, state["c"]["api"]
    if api == "evict":
        return _evict(s["ctx"], s["prob"], s)
    if api == "host":
        return _evict(s["ctx"], s["prob"], s, B.audiokv_evict_host)
    if api == "turns":  # a new prompt is described when it arrives
        return [_evict(s["ctx"], _turn_problem(s["c"], t["L"]), t) for t in s["turns"]]
    if api == "reevict":
        o = s["out"]
        B.audiokv_reevict(s["ctx"], s["prob"], s["q"], s["k"], s["v"], s["cu"], s["keep"], o["k_out"], o["v_out"],
                          o["kept_idx"], o["cu_kept"])
        return _bits({n: o[n] for n in ("k_out", "v_out", "kept_idx", "cu_kept")})
    if api == "hit":
        B.audiokv_hit_score(s["ctx"], s["attn"], s["row_len"], s["span"], s["c"]["top_k"], s["counts"], s["s_hit"])
        return {"counts": s["counts"], "s_hit": s["s_hit"]}
    ctx, prob, o = s["ctx"], s["prob"], s["out"]
    B.audiokv_score(ctx, prob, s["q"], s["k"], s["scores"])
    B.audiokv_smooth(ctx, prob, s["scores"], s["smoothed"], s["kstar"])
    B.audiokv_allocate(ctx, prob, s["S"], s["budget"], o["budgets"], o["cu_kept"])
    B.audiokv_select_gather(ctx, prob, s["smoothed"], o["budgets"], o["cu_kept"], s["k"], s["v"], o["k_out"],
                            o["v_out"], o["kept_idx"])
    B.audiokv_selection_spread(ctx, prob, o["kept_idx"], o["cu_kept"], 64, s["hist"], s["stats"])
    return dict(_bits(o), scores=s["scores"], smoothed=s["smoothed"], hist=s["hist"], stats=s["stats"])


def work(case):
    """Q and K once; of V only the rows that are kept; the kept rows and their indices out; one product Q K^T."""
    c = case
    if c["api"] == "hit":
        return {"bytes": 4 * c["heads"] * (sum(_hit_lens(c)) + 2) + 12 * c["steps"], "flops": 0}
    e = 4 if c["dtype"] == "f32" else 2
    heads, lens = c["layers"] * c["hkv"], _lens(c)
    if c["api"] == "reevict":
        kept = [c["keep"] * L for L in lens]
        rows = [b + c["new"] for b in kept]
    else:
        kept = [b / heads for b in _budgets(c, lens)]
        rows = lens
    wg = c["window"] * (c["hq"] // c["hkv"])
    total = sum(rows) * heads
    out = sum(kept) * heads
    moved = e * c["d"] * (wg * heads * len(lens) + total + 3 * out) + 4 * out + 12 * heads * len(lens)
    if c["api"] == "steps":  # the scores and the smoothed scores are outputs as well, and read by the next step
        moved += 16 * (total - heads * c["window"] * len(lens)) + 4 * out
    return {"bytes": moved, "flops": 2 * wg * c["d"] * total}


def tolerance(case):
    """Indices and rows are whole numbers; where two tokens' scores agree to fp32 rounding at a head's threshold either
    may be kept, which shifts the rows between them. Scores are fp32 sums of exponentials evaluated to 7.5e-5."""
    if case["api"] == "hit":
        return "exact"
    if case["api"] == "steps":
        return {"rel": 1e-4, "max": 4e-3, "differ": 0.01}
    return {"differ": 0.01}
