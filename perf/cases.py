"""Timed cases of the CoSA prefill path, as a program that serves or evaluates a model calls it.

A pass is one attention layer of a prefill: `cosa_kap_select` writes the visit lists, `cosa_osk_attention` walks them.
The listed cases take their shapes, budgets and planted structure from synth/configs.py where that file names them, and
otherwise stand for the ways the two calls are used: one short prompt, a fused QKV buffer, a serving engine's page pool
with prompts of different lengths, retention by Top-p, Stage 2 switched off, the library's dense path, host buffers.
"""
import math
import random

import torch

import paper_2607_25291_b200.binding as cosa

BLOCK = 128
D = 128
TILE_FLOPS = 2.0 * BLOCK * BLOCK * D     # one 128 x 128 x 128 tile product

# entry:  "lists" = KAP then OSK; "static" = the same with KAP's built-in scratch; "dense" = OSK over full lists with
#         Stage 2 off; "host" = cosa_prefill_host on pinned host buffers
# kap, osk: Stage-1 and Stage-2 budgets (osk >= 1: Stage 2 off); delta: the skip rule's scale, as a fraction of the length
BASE = {"entry": "lists", "batch": 1, "hq": 32, "hkv": 8, "n": 32768, "kap": 0.20, "osk": 0.08, "top_p": 0.0, "delta": 0.61,
        "stride": 8, "causal": True, "layout": "dense", "page": 0, "ragged": False, "band": 4, "needles": 16}


def listed():
    def case(name, **kw):
        return dict(BASE, name=name, **kw)

    return [
        # the smallest call: a short prompt of a tiny model, where the launches are what is waited for
        case("tiny_1k", hq=2, hkv=1, n=1024, kap=0.25, osk=0.10, delta=0.85, band=2, needles=2),
        # the small workload of synth/configs.py: one KV group at 4K
        case("gqa4_4k", hq=4, hkv=1, n=4096, kap=0.25, osk=0.10, delta=0.85, band=2, needles=3),
        # a request loop that may not allocate: a whole layer of a short prompt with an odd number of blocks
        case("static_31_blocks", entry="static", n=31 * BLOCK, kap=0.25, osk=0.10, delta=0.85, band=2, needles=3),
        # two prompts whose q, k, v are views into one token-major QKV buffer, odd number of blocks
        case("fused_qkv_61_blocks", batch=2, n=61 * BLOCK, kap=0.25, osk=0.10, delta=0.7, layout="fused", needles=8),
        # a serving engine's batch: 16-token pages, prompts of different lengths
        case("paged16_ragged_batch4", batch=4, n=16384, page=16, ragged=True, kap=0.20, osk=0.08, delta=0.3, needles=12),
        # the Qwen3-8B-shaped layer at 32K
        case("qwen3_32k"),
        # retention by Top-p (p = 0.95), Stage-2 budget as before, odd number of blocks
        case("topp_201_blocks", n=201 * BLOCK, kap=1.0, top_p=0.95),
        # the library's dense path: every causal block, Stage 2 off
        case("dense_16k", entry="dense", n=16384, kap=1.0, osk=1.0),
        # two cells of the Llama-3.1-8B-shaped budget sweep at 64K: Stage 2 at half of a wide Stage 1, and Stage 2 off
        case("llama31_64k_50_25", n=65536, kap=0.50, osk=0.25, delta=0.22, needles=32),
        case("llama31_64k_12_off", n=65536, kap=0.125, osk=1.0, delta=0.22, needles=32),
        # the headline workload: the Qwen3-8B-shaped layer at 128K
        case("qwen3_128k", n=131072, kap=0.10, osk=0.04, delta=0.69, needles=64),
        # the whole path on host buffers, as bench.py's end-to-end figure takes it
        case("host_16k", entry="host", n=16384, needles=8),
    ]


def draw(rng: random.Random):
    """One more case: any length from 8 to 1024 blocks, any of the options, at most the work of the 128K layer."""
    while True:
        blocks = int(round(math.exp(rng.uniform(math.log(8), math.log(1024)))))
        hq, hkv = rng.choice([(2, 1), (4, 1), (8, 8), (16, 8), (32, 8), (32, 8), (32, 4)])
        kap = rng.choice([0.05, 0.10, 0.125, 0.20, 0.25, 0.50])
        c = dict(BASE, batch=rng.choice([1, 1, 1, 2, 3]), hq=hq, hkv=hkv, n=blocks * BLOCK, kap=kap,
                 osk=round(kap * rng.choice([0.25, 0.4, 0.5]), 5), delta=round(rng.uniform(0.2, 0.85), 3),
                 stride=rng.choice([8, 8, 8, 8, 4, 16]), causal=rng.random() < 0.9, band=rng.choice([2, 4]),
                 needles=max(2, blocks // 16))
        kind = rng.choice(["plain", "plain", "plain", "fused", "paged", "topp", "off", "dense"])
        if kind == "fused":
            c["layout"] = "fused"
        elif kind == "paged":
            c["page"] = rng.choice([16, 32, 64, 128])
            c["ragged"] = c["batch"] > 1 and blocks >= 16
            if c["ragged"]:
                c["delta"] = round(c["delta"] / 2, 3)     # must stay below the shortest prompt (at least half of n)
        elif kind == "topp":
            c["kap"], c["top_p"] = 1.0, 0.95
        elif kind == "off":
            c["osk"] = 1.0
        elif kind == "dense":
            c["entry"], c["kap"], c["osk"] = "dense", 1.0, 1.0
        pairs = c["batch"] * c["hq"] * blocks * blocks * (0.5 if c["causal"] else 1.0)
        # block products of the walk, and the proxy's contraction counted in the same unit
        load = pairs * (2 * c["kap"] if c["osk"] >= 1 else (c["osk"] if c["top_p"] else c["kap"]) + c["osk"]) + pairs / c["stride"] ** 2
        limit = 32 * 1024 * 1024 * 0.5 * (0.10 + 0.04 + 1 / 64)
        if load <= limit and not (c["top_p"] and blocks > 320):
            return c


def _unit(x):
    return x / x.norm(dim=-1, keepdim=True)


def _qkv(c, gen, rng):
    """Planted structure of synth/generator.py, drawn on the GPU: a sink, a local band, needle blocks."""
    B, hq, hkv, n = c["batch"], c["hq"], c["hkv"], c["n"]
    G, nb, dev = hq // hkv, n // BLOCK, "cuda"
    if c["layout"] == "fused":
        buf = torch.empty(B, n, hq + 2 * hkv, D, dtype=torch.bfloat16, device=dev)
        q, k, v = (t.transpose(1, 2) for t in buf.split([hq, hkv, hkv], dim=2))
    else:
        q = torch.empty(B, hq, n, D, dtype=torch.bfloat16, device=dev)
        k, v = (torch.empty(B, hkv, n, D, dtype=torch.bfloat16, device=dev) for _ in range(2))
    for b in range(B):
        for g in range(hkv):
            u = _unit(torch.randn(D, generator=gen, device=dev))
            w = _unit(torch.randn(nb, D, generator=gen, device=dev))
            band = sum(torch.cat([w[m:], torch.zeros(min(m, nb), D, device=dev)])[:nb] for m in range(c["band"]))
            for h in range(g * G, (g + 1) * G):
                x = torch.randn(nb, BLOCK, D, generator=gen, device=dev)
                q[b, h] = (x + 8.0 * (u + w)[:, None, :]).view(n, D).to(torch.bfloat16)
            x = torch.randn(nb, BLOCK, D, generator=gen, device=dev) + 8.0 * band[:, None, :]
            x[0] += 10.0 * u
            k[b, g] = x.view(n, D).to(torch.bfloat16)
            v[b, g] = torch.randn(n, D, generator=gen, device=dev).to(torch.bfloat16)
            target, key = [], []
            for t in sorted(rng.sample(range(1, nb), min(c["needles"], nb - 1))):     # distinct blocks, key <= target
                free = [j for j in range(1, t + 1) if j not in key]
                target.append(t)
                key.append(rng.choice(free))
            target, key = torch.tensor(target, device=dev), torch.tensor(key, device=dev)
            mean = q[b, g * G:(g + 1) * G].reshape(G, nb, BLOCK, D).float().mean(dim=(0, 2))
            rows = (key[:, None] * BLOCK + torch.arange(BLOCK, device=dev)).reshape(-1)
            k[b, g, rows] = (0.5 * mean[target]).to(torch.bfloat16).repeat_interleave(BLOCK, 0)
    return q, k, v


def prepare(case, seed):
    c = dict(BASE, **case)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    B, hq, n, nb = c["batch"], c["hq"], c["n"], c["n"] // BLOCK
    q, k, v = _qkv(c, gen, random.Random(int(seed)))
    delta = -1.0 if c["osk"] >= 1.0 else c["delta"] * n
    s = {"case": c, "q": q, "k": k, "v": v}
    if c["entry"] == "host":
        s["shape"] = cosa.make_shape(q, k, causal=c["causal"])
        s["opt"] = cosa.default_options(stride=c["stride"], skip_scale=delta, top_p=c["top_p"])
        s["workspace"] = torch.empty(cosa.cosa_host_call_workspace_bytes(s["shape"], s["opt"]), dtype=torch.uint8, device="cuda")
        for name in ("q", "k", "v"):
            s[name] = torch.empty(s[name].shape, dtype=torch.bfloat16, pin_memory=True).copy_(s[name])
        s["out"] = torch.empty(B, hq, n, D, dtype=torch.bfloat16, pin_memory=True)
        s["lse"] = torch.empty(B, hq, n, dtype=torch.float32, pin_memory=True)
        s["visited"] = torch.empty(B, hq, nb, dtype=torch.int32, pin_memory=True)
        return s
    extra = {}
    if c["ragged"]:
        # every prompt's length: at least half of n, whole blocks
        lens = nb // 2 + 1 + torch.randint(0, nb - nb // 2, (B,), generator=gen, device="cuda")
        extra["seq_lens"] = s["lens"] = (lens * BLOCK).to(torch.int32)
    if c["page"]:
        # the sequences' pages scattered over a pool
        ps, hkv = c["page"], c["hkv"]
        pages = B * (n // ps)
        table = torch.randperm(pages, generator=gen, device="cuda").to(torch.int32).view(B, n // ps)
        for name in ("k", "v"):
            pool = torch.empty(pages, hkv, ps, D, dtype=torch.bfloat16, device="cuda")
            pool[table.view(-1).long()] = s[name].view(B, hkv, n // ps, ps, D).transpose(1, 2).reshape(pages, hkv, ps, D)
            s[name] = pool
        s["table"] = table
        extra.update(kv_page_table=table, kv_page_size=ps, kv_num_pages=pages)
    pitch = (cosa.cosa_budget_count(c["kap"], nb) + 7) // 8 * 8
    s["order"] = torch.full((B, hq, nb, pitch), -1, dtype=torch.int32, device="cuda")
    s["count"] = torch.zeros(B, hq, nb, dtype=torch.int32, device="cuda")
    if c["entry"] == "dense":
        ids = torch.arange(pitch, dtype=torch.int32, device="cuda").expand(nb, pitch)
        last = torch.arange(nb, device="cuda")[:, None] if c["causal"] else nb - 1
        s["order"][:] = torch.where(ids <= last, ids.clamp(max=nb - 1), -1)
        s["order"][..., nb:] = -1
        s["count"][:] = (torch.arange(nb, device="cuda") + 1 if c["causal"] else nb)
    s["out"] = torch.empty_like(q)
    s["lse"] = torch.empty(B, hq, n, dtype=torch.float32, device="cuda")
    s["visited"] = torch.empty(B, hq, nb, dtype=torch.int32, device="cuda")
    s["kap_opt"] = cosa.default_options(stride=c["stride"], order_stride=pitch, top_p=c["top_p"], **extra)
    s["osk_opt"] = cosa.default_options(skip_scale=delta, order_stride=pitch, **extra)
    # at start-up a program sizes the library's scratch for its longest prompt, so that calls allocate nothing
    shape = cosa.CosaShape(B, hq, c["hkv"], n, D, BLOCK, BLOCK, int(c["causal"]))
    cosa.cosa_reserve_scratch(max(cosa.cosa_workspace_bytes(0, shape, s["kap_opt"]), cosa.cosa_workspace_bytes(1, shape, s["osk_opt"])))
    return s


def run(s):
    c = s["case"]
    if c["entry"] == "host":
        cosa.cosa_prefill_host(s["q"], s["k"], s["v"], s["shape"], c["kap"], c["osk"], s["out"], s["lse"], s["visited"],
                               s["workspace"], opt=s["opt"])
        torch.cuda.current_stream().synchronize()      # the host reads the results
        return {"out": s["out"], "lse": s["lse"], "visited": s["visited"]}
    if c["entry"] == "static":
        cosa.cosa_kap_select_static(s["q"], s["k"], c["kap"], s["order"], s["count"], causal=c["causal"], opt=s["kap_opt"])
    elif c["entry"] == "lists":
        cosa.cosa_kap_select(s["q"], s["k"], c["kap"], s["order"], s["count"], causal=c["causal"], opt=s["kap_opt"])
    cosa.cosa_osk_attention(s["q"], s["k"], s["v"], s["order"], s["count"], c["osk"], s["out"], s["lse"], s["visited"],
                            causal=c["causal"], opt=s["osk_opt"])
    return {"order": s["order"], "count": s["count"], "out": s["out"], "lse": s["lse"], "visited": s["visited"]}


def work(case):
    """Each input read and each output written once; the proxy's contraction, and both products of every block the budgets
    let the walk compute (the blocks it scores beyond those depend on the values)."""
    c = dict(BASE, **case)
    B, hq, hkv, n, nb = c["batch"], c["hq"], c["hkv"], c["n"], c["n"] // BLOCK
    share = 0.75 if c["ragged"] else 1.0              # mean length of a ragged batch's prompts
    full = [int(nb * (x + 0.5) / B * 0.5 + nb * 0.5) for x in range(B)] if c["ragged"] else [nb] * B
    kept = computed = proxy = 0.0
    for m in full:
        for i in range(m):
            J = i + 1 if c["causal"] else m
            a = math.ceil(c["kap"] * J)
            b = a if c["osk"] >= 1.0 else math.ceil(c["osk"] * J)
            kept += hq * (b if c["top_p"] else a)
            computed += hq * min(a, b)
            proxy += hq * J
    rows = BLOCK // c["stride"]
    bytes_ = share * n * D * 2 * B * (2 * hq + 2 * hkv) + 4 * share * B * hq * n + 4 * B * hq * nb
    flops = 2 * TILE_FLOPS * computed
    if c["entry"] != "dense":
        bytes_ += 4 * kept + 4 * B * hq * nb          # the visit lists
        flops += proxy * 2.0 * rows * rows * D
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """P is rounded to bf16 before its product and so is the output: against the walk that keeps P in float32 and adds in
    another order, `out` differs by 2.0e-3 (largest value 0.021) and `lse` by 9e-8 on all of these; stated: four times that.
    Lists and counters are whole numbers and came out the same everywhere; a skip decision within the rounding of a float32
    logit of its threshold may fall either way."""
    return {"rel": 8e-3, "max": 8e-2, "differ": 1e-4}
