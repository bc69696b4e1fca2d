"""Workloads by which the speed of the HSA path is judged.

A case is one attention layer of one sequence: a history of `history` tokens is in the paged KV pool,
and one pass does what a generation program does per layer and query chunk through the public calls --
undo the previous pass's append (host bookkeeping only), append the chunk's K and V, select blocks,
run the forward.  `prefill` is the other direction: a whole history is appended to an empty context.

Fields of a case
    form      which calls a pass makes (see `run`)
    H, d      heads and head dimension
    chunk     tokens of the query chunk, which is also the chunk that is appended
    history   tokens in the pool after the append
    topk      blocks per head (or per head and query tile)
    ...       options of the form

Inputs are synthetic and made on the GPU from the seed: N(0, 1) queries, keys and values, or, where the
form says so, keys drawn around one mean per scene segment with the queries in an earlier segment.
"""
from __future__ import annotations

import math

import torch

from paper_2609_34606_b200 import hsa

BLOCK = 64
TILE = 128
SIGMA = 0.3       # spread of the keys around their scene segment's mean
RANK = 256        # rows a Linformer segment is compressed to
KV_BLOCKS = 195   # blocks of one KV page of the hierarchical cache: 8 frames of 1560 tokens
KV_KEEP = 4       # KV pages kept by the retrieval
TAU = (0.35, 1.0)  # threshold range of the head-adaptive selection

# Per-head budgets drawn from {0, 16, 32, 64, 128, all}: five of twelve heads look at nothing beside the
# linear branch, one at everything.
MIXED_BUDGETS = "64,0,128,64,32,0,64,32,32,-1,0,0"


def listed():
    return [
        # the smallest call: two heads of 64 over 2048 tokens -- launches and latency
        dict(name="tiny", form="step", H=2, d=64, chunk=256, history=2048, topk=4),
        # one layer of a 1.3B-class video model (12 heads of 128), 4680-token chunk, ten chunks of history
        dict(name="layer", form="step", H=12, d=128, chunk=4680, history=46800, topk=64),
        # the same layer late in a long video, pages scattered over the pool
        dict(name="long", form="step", H=12, d=128, chunk=4680, history=280800, topk=128, shuffle=True),
        # head-adaptive budgets: lists between nothing and the whole history side by side
        dict(name="budgets", form="step", H=12, d=128, chunk=4680, history=140400, topk=0, budgets=MIXED_BUDGETS,
             segment=23400),
        # one selection per 128-row query tile instead of one per head
        dict(name="tiles", form="step", H=12, d=128, chunk=4680, history=46800, topk=64, group=128),
        # the gated merge as a trained model uses it: sigmoid of one logit per token, head and dim; early
        # in a video
        dict(name="gates", form="step", H=12, d=128, chunk=4680, history=23400, topk=64, gates="dim"),
        # token-level causal: one latent frame of 1560 tokens attends to itself and what came before
        dict(name="causal", form="causal", H=12, d=128, chunk=1560, history=23400, topk=32),
        # the Linformer form of the linear branch
        dict(name="linformer", form="linformer", H=12, d=128, chunk=4680, history=46800, topk=64),
        # heads of 64, a ragged chunk, gates per token and head
        dict(name="heads64", form="step", H=16, d=64, chunk=1000, history=30000, topk=32, gates="head"),
        # hierarchical cache: retrieve KV pages, then select coarse blocks inside them; the chunk always
        # attends to itself
        dict(name="retrieve", form="retrieve", H=12, d=128, chunk=4680, history=140400, topk=32),
        # head-adaptive selection by cumulative mass over scene segments of two chunks
        dict(name="adaptive", form="adaptive", H=12, d=128, chunk=4680, history=46800, topk=0, segment=9360),
        # a history of ten chunks appended to an empty context
        dict(name="prefill", form="prefill", H=12, d=128, chunk=4680, history=46800, topk=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any form, chunks of 256 to 4680 tokens, histories of 2048 to 280,800."""
    top = max(_cost(c) for c in listed())
    while True:
        form = rng.choice(["step"] * 6 + ["causal", "linformer", "retrieve", "adaptive", "prefill", "step64"])
        d = 64 if form == "step64" else 128
        H = rng.choice([2, 4, 8, 12, 16])
        chunk = _log_int(rng, 256, 4680)
        history = max(chunk + rng.randint(1, 640), _log_int(rng, 2048, 280800))
        c = dict(form="step" if form == "step64" else form, H=H, d=d, chunk=chunk, history=history,
                 topk=_log_int(rng, 4, 128))
        if form in ("step", "step64"):
            c["gates"] = rng.choice(["", "", "head", "dim"])
            option = rng.choice(["", "", "shuffle", "group", "budgets"])
            if option == "shuffle":
                c["shuffle"] = True
            elif option == "group":
                c["group"] = rng.choice([128, 128, 256, 512])
            elif option == "budgets":
                c["topk"] = 0
                c["budgets"] = ",".join(str(rng.choice([0, 16, 32, 64, 128])) for _ in range(H - 1)) + ",-1"
                c["segment"] = max(chunk, history // rng.randint(2, 6))
        elif form == "causal":
            c["chunk"] = _log_int(rng, 256, 3120)
            c["history"] = max(c["chunk"] + rng.randint(1, 640), c["history"])
        elif form == "linformer":
            c["history"] = chunk * max(2, min(20, history // chunk))
        elif form == "retrieve":
            c["history"] = max(c["history"], 2 * KV_BLOCKS * BLOCK + rng.randint(1, 4000))
            c["topk"] = min(c["topk"], 64)
        elif form == "adaptive":
            c["topk"] = 0
            c["segment"] = max(chunk, history // rng.randint(3, 8))
        elif form == "prefill":
            c["topk"] = 0
            c["history"] = min(c["history"], 46800)
        if _cost(c) <= top and _blocks(c["history"]) <= 8192:
            return c


# ------------------------------------------------------------------ work
def _blocks(tokens):
    return (tokens + BLOCK - 1) // BLOCK


def _adaptive_blocks(case):
    """Blocks the adaptive rule keeps: nearly all of the mass lies in the queries' segment, evenly."""
    n_seg = max(1, -(-case["history"] // case["segment"]))
    tau = TAU[0] + (1.0 - 1.0 / n_seg) * (TAU[1] - TAU[0])
    return tau * case["segment"] / BLOCK


def _lists(case):
    """Selected blocks per head, one number per head."""
    n = _blocks(case["history"])
    if case.get("budgets"):
        return [n if b < 0 else min(b, n) for b in map(int, case["budgets"].split(","))]
    if case["form"] == "adaptive":
        return [min(n, _adaptive_blocks(case))] * case["H"]
    if case["form"] == "retrieve":
        own = _blocks(case["chunk"]) + 1
        return [min(n, 2 * case["topk"] + own)] * case["H"]
    return [min(n, case["topk"])] * case["H"]


def work(case):
    """Bytes (every input once, every output once) and operations of one pass."""
    H, d, Lc, N = case["H"], case["d"], case["chunk"], case["history"]
    n = _blocks(N)
    row = H * d * 2
    state = H * d * (d + 1) * 4
    if case["form"] == "prefill":
        return {"bytes": 4 * N * row + 2 * state + n * H * d * 4, "flops": 2 * N * H * d * (d + 1)}
    lists = _lists(case)
    groups = -(-Lc // case["group"]) if case.get("group") else 1
    # distinct blocks read per head: lists of several query tiles overlap as random ones do
    distinct = sum(n * (1 - (1 - k / n) ** groups) for k in lists)
    b = 4 * Lc * row + 2 * Lc * row          # append in and out, q, out
    b += H * n * d * 4                       # key sums
    b += distinct * BLOCK * d * 4            # selected K, V
    f = sum(4 * Lc * d * k * BLOCK for k in lists) + 2 * groups * n * H * d
    if case["form"] == "linformer":
        rows = (N // Lc) * RANK
        b += 2 * H * Lc * RANK * 2 + 2 * rows * row
        f += 2 * 2 * RANK * Lc * d * H + 4 * Lc * rows * d * H
    else:
        b += 3 * state
        f += 2 * 2 * Lc * H * d * (d + 1)
    if case["form"] == "causal":             # intra-chunk pairs of the linear branch
        f += 2 * H * d * Lc * (Lc + 1)
    if case.get("gates"):
        b += 2 * Lc * H * 2 * (d if case["gates"] == "dim" else 1)
    return {"bytes": int(b), "flops": int(f)}


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 250)


def tolerance(case):
    """bf16 results of sums in fp32; the lists are whole numbers that only an exact tie may change.

    Against the same path in 64 bits the outputs are off by 2.2e-3 to 2.35e-3 (2-norm) and at most by
    0.017 of their root mean square (rounding the exact result to bf16 alone: 1.7e-3 and 0.004); about
    four times that is allowed."""
    return {"rel": 1e-2, "max": 0.07, "differ": 1e-3}


# ------------------------------------------------------------------ state
def prepare(case, seed):
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    form, H, d, Lc, N = case["form"], case["H"], case["d"], case["chunk"], case["history"]
    n = _blocks(N)
    rand = lambda *shape: torch.randn(*shape, generator=g, device=dev)
    means = None
    if case.get("segment"):
        n_seg = -(-N // case["segment"])
        means = rand(n_seg, H, d)

    def keys(t0, count):
        k = rand(count, H, d)
        if means is not None:
            seg = torch.arange(t0, t0 + count, device=dev) // case["segment"]
            k = means[seg] + SIGMA * k
        return k.to(torch.bfloat16)

    lists = _lists(case)
    max_topk = n if (form == "adaptive" or case.get("budgets")) else max(1, int(max(lists)))
    opt = {}
    if form == "linformer":
        scale = Lc ** -0.5
        opt = dict(lin_mode=hsa.HSA_LIN_LINFORMER, lin_rank=RANK, lin_seg_tokens=Lc,
                   e_k=(rand(H, Lc, RANK) * scale).to(torch.bfloat16),
                   e_v=(rand(H, Lc, RANK) * scale).to(torch.bfloat16))
    order = None
    if case.get("shuffle"):
        cpu = torch.Generator()
        cpu.manual_seed(seed)
        order = torch.randperm(n, generator=cpu).to(torch.int32)
    ctx = hsa.HSAContext(H, d, max_pages=n, max_q_tokens=Lc, max_topk=max_topk, page_order=order, device=dev,
                         causal=form == "causal", adaptive=form == "adaptive",
                         gate_act=1 if case.get("gates") else 0, **opt)
    s = {"case": dict(case), "ctx": ctx}
    if form == "prefill":
        s["k"], s["v"] = keys(0, N), rand(N, H, d).to(torch.bfloat16)
        return s
    n0 = N - Lc
    t = 0
    while t < n0:
        m = min(Lc, n0 - t)
        ctx.append_kv(keys(t, m), rand(m, H, d).to(torch.bfloat16))
        t += m
    s["n0"] = n0
    s["k"], s["v"] = keys(n0, Lc), rand(Lc, H, d).to(torch.bfloat16)
    q = rand(Lc, H, d)
    if means is not None:
        q = means[seed % max(1, means.shape[0] - 1)] + SIGMA * q
    s["q"] = q.to(torch.bfloat16)
    s["out"] = torch.empty_like(s["q"])
    if form != "adaptive":
        budgets = [int(b) for b in case["budgets"].split(",")] if case.get("budgets") else [case["topk"]] * H
        s["budgets"] = torch.tensor(budgets, dtype=torch.int32, device=dev)
        s["sel"] = ctx.alloc_selection(Lc, case.get("group", 0))
    if case.get("gates"):
        shape = (Lc, H, d) if case["gates"] == "dim" else (Lc, H)
        s["g_lin"], s["g_sp"] = rand(*shape).to(torch.bfloat16), rand(*shape).to(torch.bfloat16)
    return s


def _pages(pool, ctx):
    return pool.view(torch.bfloat16).view(ctx.max_pages, ctx.H, BLOCK, ctx.d)


def run(s):
    case, ctx = s["case"], s["ctx"]
    form, Lc, N = case["form"], case["chunk"], case["history"]
    if form == "prefill":
        ctx.rewind(0)
        ctx.state.zero_()
        for t in range(0, N, Lc):
            ctx.append_kv(s["k"][t:t + Lc], s["v"][t:t + Lc])
        return {"k": _pages(ctx.k_pool, ctx), "v": _pages(ctx.v_pool, ctx), "ksum": ctx.ksum, "S": ctx.S, "z": ctx.z}
    ctx.rewind(s["n0"])
    ctx.append_kv(s["k"], s["v"])
    res = {}
    q, causal, group = s["q"], form == "causal", case.get("group", 0)
    pos = s["n0"] if causal else N
    if form == "adaptive":
        idx, cnt, res["gini_tau"] = ctx.select_blocks_adaptive(q, *TAU)
    elif form == "retrieve":
        kept = ctx.retrieve_kv_pages(q, KV_BLOCKS, KV_KEEP)
        idx, cnt = ctx.select_blocks_ex(q, s["budgets"], 2, s["n0"] // BLOCK, None, sel=s["sel"], kv_pages=kept,
                                        kv_page_blocks=KV_BLOCKS)
        res["kept"] = kept
    else:
        idx, cnt = ctx.select_blocks(q, s["budgets"], q_pos0=pos, causal=causal, group_tokens=group, sel=s["sel"])
    ctx.forward(q, idx, cnt, q_pos0=pos, causal=causal, group_tokens=group, g_lin=s.get("g_lin"), g_sp=s.get("g_sp"),
                out=s["out"])
    res.update(out=s["out"], idx=idx, cnt=cnt, ksum=ctx.ksum, k=_pages(ctx.k_pool, ctx), v=_pages(ctx.v_pool, ctx))
    if form == "linformer":
        rows = ctx.n_tokens // Lc * RANK // BLOCK
        res["k_compressed"] = ctx.kc_pool.view(torch.bfloat16).view(-1, ctx.H, BLOCK, ctx.d)[:rows]
        res["v_compressed"] = ctx.vc_pool.view(torch.bfloat16).view(-1, ctx.H, BLOCK, ctx.d)[:rows]
    else:
        res["S"], res["z"] = ctx.S, ctx.z
    return res
