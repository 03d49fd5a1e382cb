"""The work a user of this library has it do, as cases that can be timed: what each one stands for, its inputs, one
pass through the public entry points, the bytes and operations the pass cannot do without.

Inputs: Gaussian queries, keys and values in which every key also carries its own share of a direction the window
queries have in common (the vertical stripes of real attention maps: the same keys matter to all window rows), a few
planted needle keys and attention-sink keys; budgets from a heavy-tailed INF_sc table.
"""
import math

import torch

from paper_2508_15806_b200 import binding as B
from paper_2508_15806_b200 import context_parallel as CP

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


# ---- the cases ---------------------------------------------------------------------------------------------------
def _case(kind, **kw):
    """Defaults: a Llama-3-8B / Mistral-7B layer (32 query heads, 8 KV heads, head_dim 128, bf16, window 32, pool 7)."""
    c = dict(kind=kind, n_layers=1, n_q_heads=32, n_kv_heads=8, head_dim=128, dtype="bf16", window=32, pool=7,
             pool_avg=False, all_causal=False, lse=False, n_seqs=1, len_min=8192, len_max=8192, avg_budget=512,
             fixed=64, skew="lognormal")
    c.update(kw)
    return c


def listed():
    return [
        # Stage 2 of the method, once per model: 32 layers x 8 KV heads
        dict(name="budgets", kind="alloc", n_layers=32, n_heads=8, fixed=64, avg_budget=512, within_layer=False, cap=0),
        # Stage 1, calibration: the heads of 32 layers x 32 heads over eight probe prompts of 4096 tokens
        dict(name="behaviour", kind="behavior", n_rows=8192, row_len=4096, n_needle=12, top_k=16),
        # the smallest compression: one fp32 multi-head layer of 1024 tokens, one call, latency counts
        _case("layer", name="layer-f32-1k", n_q_heads=8, head_dim=64, dtype="f32", window=16, pool=5, len_min=1024,
              len_max=1024, avg_budget=128, fixed=32),
        # an ordinary call: one bf16 layer of 8192 tokens
        _case("layer", name="layer-8k"),
        # scores alone (head_dim 64, odd length, mean pooling, the prefill attention's own softmax domain)
        _case("score", name="score-d64-4k", head_dim=64, pool=5, pool_avg=True, all_causal=True, len_min=4093,
              len_max=4093),
        # a short prompt through the whole model: 32 layers, issue rate and launches count
        _case("model", name="model-4k", n_layers=32, len_min=4001, len_max=4001, avg_budget=256),
        # the 32k-context model step
        _case("model", name="model-32k", n_layers=32, len_min=32768, len_max=32768),
        # the same behind a prefill attention that hands its row statistics over (one pass over the keys)
        _case("model", name="model-32k-lse", n_layers=32, len_min=32768, len_max=32768, lse=True),
        # a batch of eight ragged prompts, window 64
        _case("model", name="model-batch", n_layers=32, window=64, n_seqs=8, len_min=4096, len_max=32768,
              avg_budget=1024),
        # long context: 131072 tokens, window 64, a few heads take most of the budget
        _case("model", name="model-128k", n_layers=32, window=64, len_min=131072, len_max=131072, avg_budget=4096,
              skew="extreme"),
        # tensors in host memory (pinned): copies in and out are part of the call
        _case("host", name="host-32k", len_min=32768, len_max=32768),
        # one rank's share of a sequence split over ranks: the context-parallel call sequence
        _case("shard", name="shard-32k", window=64, len_min=32768, len_max=32768, avg_budget=1024),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["alloc", "behavior", "layer", "layer", "score", "model", "model", "model", "host", "shard"])
    if kind == "alloc":
        fixed, avg = rng.choice([0, 32, 64]), _log_int(rng, 128, 4096)
        return dict(kind=kind, n_layers=_log_int(rng, 8, 96), n_heads=rng.choice([1, 2, 4, 8, 16, 32]), fixed=fixed,
                    avg_budget=avg, within_layer=rng.random() < 0.3, cap=rng.choice([0, 0, 4 * avg]))
    if kind == "behavior":
        return dict(kind=kind, n_rows=_log_int(rng, 64, 16384), row_len=_log_int(rng, 1024, 6144),
                    n_needle=rng.randint(4, 48), top_k=rng.randint(8, 48))
    avg = _log_int(rng, 128, 2048)
    if kind in ("layer", "score"):
        f32 = rng.random() < 0.35
        top = _log_int(rng, 512, 6000 if f32 else 16384)
        c = _case(kind, dtype="f32" if f32 else "bf16", head_dim=rng.choice([64, 128]), n_q_heads=rng.choice([8, 16, 32]),
                  window=rng.choice([16, 32]), pool=rng.choice([5, 7]), pool_avg=rng.random() < 0.3,
                  all_causal=rng.random() < 0.3, n_seqs=rng.choice([1, 1, 2, 5]), len_max=top,
                  len_min=max(300, top // rng.choice([1, 2, 4])), avg_budget=min(avg, 512))
        c["len_min"] = min(c["len_min"], c["len_max"])
        return c
    if kind == "model":
        n_seqs = rng.choice([1, 1, 2, 4, 8])
        top = _log_int(rng, 2000, 131072 // n_seqs)
        return _case(kind, n_layers=rng.randint(8, 32), window=rng.choice([16, 32, 64]), n_seqs=n_seqs, len_max=top,
                     len_min=top // 2 if n_seqs > 1 else top, avg_budget=avg, lse=rng.random() < 0.3,
                     skew=rng.choice(["lognormal", "extreme"]))
    top = _log_int(rng, 4096, 40000)
    return _case(kind, window=rng.choice([32, 64]), len_min=top, len_max=top, avg_budget=avg)


# ---- sizes that follow from a case ---------------------------------------------------------------------------------
def _lens(c):
    """Sequence lengths of the case: evenly spread over [len_min, len_max] in a fixed shuffled order, odd ones among
    them."""
    n = c["n_seqs"]
    if n == 1:
        return [c["len_max"]]
    step = (c["len_max"] - c["len_min"]) / (n - 1)
    return [int(c["len_min"] + step * ((3 * i + 1) % n)) for i in range(n)]


def _cu(c):
    cu = [0]
    for n in _lens(c):
        cu.append(cu[-1] + n)
    return cu


def _n_hist(c):
    return sum(max(n - c["window"], 0) for n in _lens(c))


def _rows(c, budgets_row):
    return sum(min(n, max(int(b), c["window"])) for n in _lens(c) for b in budgets_row)


# ---- inputs ---------------------------------------------------------------------------------------------------------
def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFF)
    return g


def _inf_sc(g, n_layers, n_heads, skew):
    """INF_sc per (layer, head): lognormal, or near zero for all but six heads."""
    t = torch.randn(n_layers, n_heads, generator=g, device="cuda")
    if skew == "extreme":
        t = 1e-4 * torch.exp(0.5 * t)
        heavy = torch.randint(0, n_layers * n_heads, (6,), generator=g, device="cuda")
        t.view(-1)[heavy] = 1.0
        return t.contiguous()
    return torch.exp(1.5 * t).contiguous()


def _qkv(c, g):
    """One layer's q_win [n_seqs, w, Hq, d], k, v [T, Hkv, d]."""
    dt, d, w = DTYPES[c["dtype"]], c["head_dim"], c["window"]
    hq, hkv, cu = c["n_q_heads"], c["n_kv_heads"], _cu(c)
    T, n, G = cu[-1], c["n_seqs"], hq // hkv
    q = torch.randn(n, w, hq, d, generator=g, device="cuda", dtype=dt)
    k = torch.randn(T, hkv, d, generator=g, device="cuda", dtype=dt)
    v = torch.randn(T, hkv, d, generator=g, device="cuda", dtype=dt)
    u = torch.randn(n, hkv, d, generator=g, device="cuda")
    u = u / u.norm(dim=2, keepdim=True)
    gain = 4.0
    q += (gain * u).repeat_interleave(G, dim=1).unsqueeze(1).to(dt)
    # a key's share of the common direction: logits of standard deviation 1.5; needles 8 and sinks 6 above the rest
    amp = torch.randn(T, hkv, generator=g, device="cuda") * 1.5
    for s in range(n):
        n_hist = cu[s + 1] - cu[s] - w
        if n_hist > 64:
            amp[cu[s]:cu[s] + 4] += 6.0
            at = torch.randint(4, n_hist, (16,), generator=g, device="cuda") + cu[s]
            amp[at] += 8.0
        part = (amp[cu[s]:cu[s + 1]] * (math.sqrt(d) / gain)).to(dt)
        k[cu[s]:cu[s + 1]].addcmul_(part.unsqueeze(2), u[s].to(dt).unsqueeze(0))
    return q, k, v


def _params(c, q, k, v):
    return B.make_params(q, k, v, c["window"], c["pool"], B.SLKV_POOL_AVG if c["pool_avg"] else B.SLKV_POOL_MAX,
                         softmax_domain=B.SLKV_ALL_CAUSAL if c["all_causal"] else B.SLKV_HISTORY)


def prepare(case, seed):
    c, g = case, _gen(seed)
    if c["kind"] == "alloc":
        opt = None
        if c["within_layer"] or c["cap"]:
            opt = B.SlkvAllocOptions(B.SLKV_NORM_WITHIN_LAYER if c["within_layer"] else B.SLKV_NORM_GLOBAL,
                                     B.SLKV_ROUND_SUM_EXACT, c["cap"])
        return dict(case=c, inf=_inf_sc(g, c["n_layers"], c["n_heads"], "lognormal"), options=opt,
                    total=c["n_layers"] * c["n_heads"] * c["avg_budget"],
                    budgets=torch.empty(c["n_layers"], c["n_heads"], dtype=torch.int32, device="cuda"),
                    status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if c["kind"] == "behavior":
        # rows of attention weights: a sink, a needle span with a share of the mass (small for most heads), background
        n, L, m = c["n_rows"], c["row_len"], c["n_needle"]
        a = torch.exp(0.7 * torch.randn(n, L, generator=g, device="cuda"))
        start = 1 + (torch.rand(n, 1, generator=g, device="cuda") * (L - m - 1)).long()
        needle = start + torch.arange(m, device="cuda").unsqueeze(0)
        share = torch.rand(n, 1, generator=g, device="cuda") ** 3
        a.mul_(0.7 * (1 - share) / a.sum(dim=1, keepdim=True))
        a[:, :1] += 0.3 * (1 - share)
        wn = torch.exp(1.2 * torch.randn(n, m, generator=g, device="cuda"))
        a.scatter_add_(1, needle, wn / wn.sum(dim=1, keepdim=True) * share)
        top = torch.topk(a, c["top_k"], dim=1).indices
        return dict(case=c, attn=a, needle=needle.int().contiguous(), topk=top.int().contiguous())

    # a model's table is its own whatever the prompt: the same budgets, and so the same output sizes, for every seed
    inf = _inf_sc(_gen(0), c["n_layers"], c["n_kv_heads"], c["skew"])
    total = c["n_layers"] * c["n_kv_heads"] * c["avg_budget"]
    budgets = B.slkv_alloc_budgets(inf, c["fixed"], total)
    cu, w, d, dt = _cu(c), c["window"], c["head_dim"], DTYPES[c["dtype"]]
    layers = [_qkv(c, _gen(seed, 1 + l)) for l in range(c["n_layers"])]
    p = _params(c, *layers[0])
    st = dict(case=c, cu=cu, params=p, layers=layers, budgets=[budgets[l].contiguous() for l in range(c["n_layers"])])
    rows = [_rows(c, r) for r in budgets.tolist()]
    n_seg = c["n_seqs"] * c["n_kv_heads"]
    if c["kind"] == "shard":
        q, k, v = layers[0]
        st["shard"] = CP.shard_of(q, k, v, w, c["pool"], 0, 1)
        st["comm"] = _OneRank()
        return st
    if c["kind"] == "host":
        pin = lambda t: t.cpu().pin_memory()                                                        # noqa: E731
        st["layers"] = [tuple(pin(t) for t in x) for x in layers]
        st["budgets"] = [b.cpu() for b in st["budgets"]]
        st["out"] = [torch.empty(rows[0], d, dtype=dt).pin_memory(), torch.empty(rows[0], d, dtype=dt).pin_memory(),
                     torch.empty(n_seg + 1, dtype=torch.int32).pin_memory(),
                     torch.empty(rows[0], dtype=torch.int32).pin_memory()]
        st["arena"] = torch.empty(B.slkv_compress_host_arena_bytes(p, cu, rows[0]), dtype=torch.uint8, device="cuda")
        return st
    st["cu_dev"] = torch.tensor(cu, dtype=torch.int32, device="cuda")
    st["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    many = c["kind"] == "model"
    n_ws = B.slkv_workspace_bytes_overlapped(p, cu) if many else B.slkv_workspace_bytes(p, cu)
    st["ws"] = torch.empty(n_ws, dtype=torch.uint8, device="cuda")
    if c["kind"] == "score":
        st["pooled"] = torch.zeros(B.slkv_pooled_elems(p, cu), dtype=torch.float32, device="cuda")
        return st
    # the packed cache of all layers: one allocation, a slice for each layer
    first = [0]
    for r in rows:
        first.append(first[-1] + r)
    st["k_out"] = torch.zeros(first[-1], d, dtype=dt, device="cuda")
    st["v_out"] = torch.zeros(first[-1], d, dtype=dt, device="cuda")
    st["kept"] = torch.zeros(first[-1], dtype=torch.int32, device="cuda")
    st["offsets"] = torch.zeros(c["n_layers"], n_seg + 1, dtype=torch.int32, device="cuda")
    st["slices"] = [(st["k_out"][a:b], st["v_out"][a:b], st["offsets"][l], st["kept"][a:b])
                    for l, (a, b) in enumerate(zip(first, first[1:]))]
    st["lse"] = [None] * c["n_layers"]
    if c["lse"]:
        for l, (q, k, _) in enumerate(layers):
            st["lse"][l] = torch.zeros(c["n_seqs"], c["n_q_heads"], w, dtype=torch.float32, device="cuda")
            B.slkv_row_lse(p, q, k, st["cu_dev"], cu, st["lse"][l], st["ws"])
    return st


class _OneRank:
    """The communicator of a job of one rank."""
    rank, world = 0, 1

    def all_gather(self, t):
        return t.unsqueeze(0)

    def all_reduce_sum(self, t):
        return t


# ---- one pass -------------------------------------------------------------------------------------------------------
def _bits(t):
    """Packed rows are bit copies of input rows: compared as whole values."""
    return t.view(torch.int16 if t.element_size() == 2 else torch.int32)


def run(state):
    s = state
    c = s["case"]
    kind = c["kind"]
    if kind == "alloc":
        return B.slkv_alloc_budgets(s["inf"], c["fixed"], s["total"], s["budgets"], s["status"], options=s["options"])
    if kind == "behavior":
        return B.slkv_behavior_scores(s["attn"], s["needle"], s["topk"])
    p, cu = s["params"], s["cu"]
    if kind == "shard":
        o = CP.compress_rank(s["shard"], s["budgets"][0], c["pool"], s["comm"])
        return [_bits(o["k_out"]), _bits(o["v_out"]), o["offsets"], o["kept_idx"], o["pooled"], o["lse"]]
    if kind == "host":
        q, k, v = s["layers"][0]
        k_out, v_out, offsets, kept = s["out"]
        n = B.slkv_compress_host(p, q, k, v, cu, s["budgets"][0], k_out, v_out, offsets, kept, s["arena"])
        return [_bits(k_out), _bits(v_out), offsets, kept, n]
    if kind == "score":
        q, k, _ = s["layers"][0]
        return B.slkv_score(p, q, k, s["cu_dev"], cu, s["pooled"], s["ws"], s["status"])
    call = B.slkv_compress if kind == "layer" else B.slkv_compress_overlapped
    for (q, k, v), bud, (k_out, v_out, offsets, kept), lse in zip(s["layers"], s["budgets"], s["slices"], s["lse"]):
        call(p, q, k, v, s["cu_dev"], cu, bud, k_out, v_out, offsets, kept, s["ws"], None, s["status"], lse=lse)
    if kind == "model":
        B.slkv_join()
    return [_bits(s["k_out"]), _bits(s["v_out"]), s["offsets"], s["kept"], s["status"]]


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def work(case):
    c = case
    if c["kind"] == "alloc":
        n = c["n_layers"] * c["n_heads"]
        return {"bytes": 8 * n, "flops": 8 * n}
    if c["kind"] == "behavior":
        per_row = 8 * (c["n_needle"] + c["top_k"]) + 12                  # indices, the weights at them, three scores
        return {"bytes": c["n_rows"] * per_row, "flops": c["n_rows"] * (c["n_needle"] + c["top_k"])}
    e = 4 if c["dtype"] == "f32" else 2
    d, hkv, nl, T = c["head_dim"], c["n_kv_heads"], c["n_layers"], sum(_lens(c))
    n_hist = _n_hist(c)
    # one product of the window queries with every history key (two where the row statistics are not given)
    passes = 1 if c["lse"] else 2
    flops = passes * 2.0 * c["n_q_heads"] * c["window"] * n_hist * d
    nbytes = hkv * T * d * e + c["n_seqs"] * c["window"] * c["n_q_heads"] * d * e
    if c["kind"] == "score":
        return {"bytes": nbytes + 4 * hkv * n_hist, "flops": flops}
    # kept rows of K and V read and written once (K's were read above); the average budget bounds what is kept
    kept = min(hkv * c["avg_budget"] * c["n_seqs"], hkv * T)
    out = kept * (3 * d * e + 4)
    if c["kind"] == "shard":                                             # capacity rows are cleared and returned whole
        out = hkv * T * (2 * d * e + 4) + kept * d * e + 4 * hkv * n_hist
    return {"bytes": nl * (nbytes + out), "flops": nl * flops}


def tolerance(case):
    """Scores: fp32 sums of a few hundred exponentials; ratios of fp64 sums come back in fp32.  Kept positions and the
    rows copied for them: whole values, the same but for ties within the scores' rounding at a head's last place."""
    if case["kind"] == "alloc":
        return "exact"
    if case["kind"] == "behavior":
        return {"rel": 1e-6}
    return {"rel": 2e-5, "differ": 0.01}
