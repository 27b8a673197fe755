"""The work that is measured: verification steps, prompt prefills and the stand-alone linear layer,
each through the entry point a program calls, at the repository's own model shapes.

A step's cost is a fixed part plus an equal part for every active layer, so most cases run a
decoder cut to a few layers (embedding, layers, final norm, LM head and acceptance all included);
one runs the whole 7B shape.

Weights are drawn like a trained decoder's where it matters to the path: projections N(0, 0.02),
residual outputs scaled by 1/sqrt(2 L), gains around one, and an LM head that prefers three
successors of every token (a bigram), so that drafts are accepted in part, distributions are
peaked, and tokens do not hang on the last bits of a logit.
"""
import dataclasses
import math

import torch

from paper_2609_26100_gb300 import native, synth
from paper_2609_26100_gb300.runner import TssRunner

MODELS = {"tiny": synth.TINY, "7b": synth.LLAMA2_7B, "13b": synth.LLAMA2_13B}
STRIDE = 64  # path columns of the result arrays
BOOST = (20.0, 19.0, 18.0)  # logits a token's three successors gain


def listed():
    return [
        # the smallest call: the tiny decoder's chain, where launches and latency are all there is
        {"name": "tiny_chain", "kind": "verify", "model": "tiny", "layers": 4, "skips": "2", "ctx": "128",
         "block": "chain", "k": 4, "mode": "greedy", "host": False},
        # the same for a caller that keeps tokens and results in pinned host memory
        {"name": "tiny_batch_host", "kind": "verify", "model": "tiny", "layers": 4, "skips": "2;0,3", "ctx": "97,255,31,512",
         "block": "chain", "k": 7, "mode": "greedy", "host": True},
        # the headline: one user's chain on the whole 7B model, 4 of 32 layers skipped
        {"name": "7b_chain", "kind": "verify", "model": "7b", "layers": 32, "skips": "20,24,27,30", "ctx": "1024",
         "block": "chain", "k": 5, "mode": "greedy", "host": False},
        # a 60-node draft tree
        {"name": "7b_tree", "kind": "verify", "model": "7b", "layers": 4, "skips": "2", "ctx": "2048",
         "block": "eagle", "k": 60, "mode": "greedy", "host": False},
        # a wide static tree (127 nodes) at an odd context
        {"name": "7b_wide_tree", "kind": "verify", "model": "7b", "layers": 2, "skips": "", "ctx": "777",
         "block": "wide", "k": 127, "mode": "greedy", "host": False},
        # a serving batch: 24 users, ragged contexts, short chains
        {"name": "7b_batch", "kind": "verify", "model": "7b", "layers": 4, "skips": "1;3",
         "ctx": "113,1450,700,64,2047,389,901,1200,256,33,811,1620,540,77,1333,462,1019,205,1777,620,948,1501,350,128",
         "block": "chain", "k": 5, "mode": "greedy", "host": False},
        # long contexts: 16 users, bound by the KV cache
        {"name": "7b_long", "kind": "verify", "model": "7b", "layers": 4, "skips": "2",
         "ctx": ",".join(["16384"] * 16), "block": "chain", "k": 8, "mode": "greedy", "host": False},
        # mixed domains and ragged contexts on the 13B shape, speculative sampling
        {"name": "13b_mixed_sample", "kind": "verify", "model": "13b", "layers": 4, "skips": "1;3;0,2;2;1,3;0",
         "ctx": "644,3059,1907,2511,812,4001,1333,2250", "block": "chain", "k": 5, "mode": "sample", "host": False},
        # the same batch verified group by group (one step per skip set)
        {"name": "13b_grouped", "kind": "grouped", "model": "13b", "layers": 4, "skips": "1;3;0,2",
         "ctx": "644,3059,1907,2511,812,4001", "block": "chain", "k": 5, "mode": "greedy", "host": False},
        # prompts: four of 1024 tokens at once, and one short one appended to a conversation
        {"name": "7b_prefill_4x1024", "kind": "prefill", "model": "7b", "layers": 4, "skips": "2", "ctx": "0,0,0,0",
         "tokens": "1024,1024,1024,1024"},
        {"name": "7b_prefill_200", "kind": "prefill", "model": "7b", "layers": 4, "skips": "2", "ctx": "333",
         "tokens": "200"},
        # the linear layer on its own: the fused QKV projection of six rows
        {"name": "linear_6x4096x12288", "kind": "linear", "rows": 6, "k_dim": 4096, "n_out": 12288},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["verify", "verify", "verify", "tree", "sample", "grouped", "prefill", "prefill", "linear"])
    if kind == "linear":
        return {"kind": "linear", "rows": log_int(1, 64), "k_dim": 64 * log_int(4, 220), "n_out": 128 * log_int(2, 96)}
    model = rng.choice(["tiny", "7b", "7b", "13b"])
    layers = rng.randint(2, 4)
    # layer `layers - 1` is never skipped by the first domain, so every batch runs something
    skips = [",".join(str(x) for x in sorted(rng.sample(range(layers - 1), rng.randint(0, min(2, layers - 1)))))
             for _ in range(rng.randint(1, 3))]
    case = {"kind": "verify" if kind in ("tree", "sample") else kind, "model": model, "layers": layers,
            "skips": ";".join(skips)}
    if kind == "prefill":
        n = rng.choice([1, 1, 2, 4])
        return {**case, "ctx": ",".join(str(rng.choice([0, log_int(1, 1500)])) for _ in range(n)),
                "tokens": ",".join(str(log_int(8, 1024)) for _ in range(n))}
    if kind == "tree":
        n, block, k = rng.choice([1, 1, 2]), rng.choice(["eagle", "wide"]), log_int(8, 63)
        if block == "wide" and n == 1:
            k = log_int(24, 127)
    else:
        block, k = "chain", rng.randint(1, 9)
        n = min(log_int(1, 48), 256 // (k + 1))
    top = min(16384, 130000 // n)
    return {**case, "ctx": ",".join(str(log_int(8, top)) for _ in range(n)), "block": block, "k": k,
            "mode": "sample" if kind == "sample" else "greedy", "host": kind != "grouped" and rng.random() < 0.25}


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def arch_of(case):
    return dataclasses.replace(MODELS[case["model"]], n_layers=case["layers"])


def ints(text):
    return [int(x) for x in text.split(",") if x]


def masks_of(case):
    """The skip bitmask of every domain."""
    return [sum(1 << l for l in ints(s)) for s in case["skips"].split(";")]


def domains_of(case):
    n = len(ints(case["ctx"]))
    return [b % len(masks_of(case)) for b in range(n)]


def parents_of(case):
    if case["kind"] == "prefill":
        return [synth.chain_parents(n - 1) for n in ints(case["tokens"])]
    if case["block"] == "chain":
        one = synth.chain_parents(case["k"])
    elif case["block"] == "eagle":
        one = synth.eagle_tree(case["k"], (4, 3, 2, 2, 1, 1))
    else:
        one = synth.eagle_tree(case["k"], (8, 4, 3, 2, 2, 1, 1, 1))
    return [one] * len(ints(case["ctx"]))


class Source:
    """Seeded normal and integer tensors on the GPU, one stream for every tag."""

    def __init__(self, seed):
        self.seed = seed

    def gen(self, tag):
        return torch.Generator("cuda").manual_seed((self.seed * 1000003 + tag * 7919) % (1 << 62))

    def normal(self, tag, shape, std=1.0, mean=0.0):
        return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(mean, std, generator=self.gen(tag))

    def ints(self, tag, n, high):
        return torch.randint(0, high, (n,), generator=self.gen(tag), device="cuda")


def layer_weights(src, arch, l):
    d, f, r = arch.d_model, arch.d_mlp, 0.02 / math.sqrt(2 * arch.n_layers)
    t = 100 + 16 * l
    return {"attn_norm": src.normal(t, (d,), 0.1, 1.0), "wq": src.normal(t + 1, (d, d), 0.02),
            "wk": src.normal(t + 2, (d, d), 0.02), "wv": src.normal(t + 3, (d, d), 0.02),
            "wo": src.normal(t + 4, (d, d), r), "mlp_norm": src.normal(t + 5, (d,), 0.1, 1.0),
            "w_gate": src.normal(t + 6, (f, d), 0.02), "w_up": src.normal(t + 7, (f, d), 0.02),
            "w_down": src.normal(t + 8, (d, f), r)}


def ends(src, arch):
    """Embedding, LM head, final gain and the three successors of every token."""
    V, d = arch.vocab, arch.d_model
    embed, head = src.normal(1, (V, d)), src.normal(2, (V, d), 0.02)
    order = torch.randperm(V, generator=src.gen(3), device="cuda")
    place = torch.empty_like(order)
    place[order] = torch.arange(V, device="cuda")
    nxt = torch.stack([order[(place + j) % V] for j in (1, 2, 3)])  # [3][V]
    w = head.float()
    for j, boost in enumerate(BOOST):  # (a residual stream's cosine with its embedding is about 0.6)
        w[nxt[j]] += boost / (0.6 * d) * embed.float()
    return embed, w.to(torch.bfloat16), src.normal(4, (d,), 0.1, 1.0), nxt


def context(src, arch, l, b, n):
    """The cached K and V of one request's context in one layer."""
    return src.normal(5000 + 64 * l + b, (2, arch.n_heads, n, arch.head_dim))


def block_tokens(src, case, arch, nxt):
    """Every request's block, concatenated: drafts that follow the bigram for the most part; with
    sampling, the draft distributions they were drawn from too."""
    par = parents_of(case)
    V, M = arch.vocab, sum(len(p) for p in par)
    tok = src.ints(6, M, V)
    if case["kind"] == "prefill":
        return tok.to(torch.int32), None
    first = [0]
    for p in par:
        first.append(first[-1] + len(p))
    depth = [d for p in par for d in synth.depths_of(p)]
    up = [first[b] + i for b, p in enumerate(par) for i in p]  # parent row (roots: unused)
    rank = [0] * M  # a node's place among its siblings
    kids = {}
    for m in range(M):
        if depth[m]:
            rank[m] = kids.get(up[m], 0)
            kids[up[m]] = rank[m] + 1
    follow = (torch.rand(M, generator=src.gen(7), device="cuda") < 0.9).tolist()
    probs = torch.empty((M, V), dtype=torch.float32, device="cuda") if case["mode"] == "sample" else None
    if probs is not None:
        probs.normal_(generator=src.gen(8))
        noise = torch.empty((M, V), dtype=torch.float32, device="cuda").exponential_(generator=src.gen(9))
    for t in range(1, max(depth) + 1):
        rows = [m for m in range(M) if depth[m] == t]
        above = tok[torch.tensor([up[m] for m in rows], device="cuda")]
        if probs is not None:
            i = torch.tensor(rows, device="cuda")
            for j, boost in enumerate((18.0, 17.5, 17.0)):
                probs[i, nxt[j][above]] += boost
            tok[i] = (torch.softmax(probs[i].double(), -1) / noise[i]).argmax(-1)
        else:
            use = [(m, j) for j, m in enumerate(rows) if follow[m] and rank[m] < 3]
            if use:
                i, j = torch.tensor(use, device="cuda").T
                tok[i] = nxt[torch.tensor([rank[m] for m, _ in use], device="cuda"), above[j]]
    return tok.to(torch.int32), None if probs is None else torch.softmax(probs.double(), -1).float()


def prepare(case, seed):
    src = Source(seed)
    if case["kind"] == "linear":
        x, w = src.normal(1, (case["rows"], case["k_dim"])), src.normal(2, (case["n_out"], case["k_dim"]), 0.02)
        return {"case": case, "x": x, "w": w,
                "y": torch.zeros((case["rows"], case["n_out"]), dtype=torch.float32, device="cuda")}
    arch, ctx, masks, doms, par = arch_of(case), ints(case["ctx"]), masks_of(case), domains_of(case), parents_of(case)
    embed, head, gain, nxt = ends(src, arch)
    weights = {"embed": embed, "lm_head": head, "final_norm": gain,
               "layers": [layer_weights(src, arch, l) for l in range(arch.n_layers)]}
    union = [l for l in range(arch.n_layers) if any(not (masks[d] >> l) & 1 for d in doms)]
    prefill = case["kind"] == "prefill"
    rows = [len(p) for p in par]
    run = TssRunner(arch, weights, n_slots=len(ctx), kv_cap=max(c + n for c, n in zip(ctx, rows)) + 8,
                    max_batch=len(ctx), max_rows=256 if prefill else max(16, sum(rows)),
                    max_nodes=64 if prefill else max(rows), kv_layers=union)
    del weights, embed, head
    run.set_phi(dict(enumerate(masks)))
    for b, c in enumerate(ctx):
        for l in union:
            if c and not (masks[doms[b]] >> l) & 1:
                run.kv[l][b, :, :, :c] = context(src, arch, l, b, c)
    tok, probs = block_tokens(src, case, arch, nxt)
    state = {"case": case, "run": run, "kv": [run.kv[l] for l in union]}
    if prefill:
        state["prompts"], at = [], 0
        for n in rows:
            state["prompts"].append(tok[at:at + n].tolist())
            at += n
    else:
        host = case["host"]
        if host:
            tok = tok.cpu().pin_memory()
            probs = None if probs is None else probs.cpu().pin_memory()
        reqs = [synth.Request(c, p, [], d) for c, p, d in zip(ctx, par, doms)]
        state["batch"] = run.batch(reqs, tokens=tok, mode=native.TSS_MODE_SAMPLE if case["mode"] == "sample" else native.TSS_MODE_GREEDY,
                                   draft_probs=probs, philox_seed=seed, io_host=host)
        state["res"] = run.alloc_results(len(ctx), sum(rows), path_stride=STRIDE, host=host)
    torch.cuda.empty_cache()
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "linear":
        native.linear_static(state["x"], state["w"], state["y"], torch.cuda.current_stream().cuda_stream)
        return state["y"]
    r = state["run"]
    if case["kind"] == "prefill":
        r.prefill(state["prompts"], ints(case["ctx"]), domains_of(case))
        return {"kv": state["kv"]}
    res = state["res"]
    (r.verify_grouped if case["kind"] == "grouped" else r.verify)(state["batch"], res)
    return {"logits": res["logits"], "accept_len": res["accept_len"], "bonus": res["bonus"], "path": res["path"],
            "new_ctx_len": res["new_ctx_len"], "kv": state["kv"]}


def work(case):
    if case["kind"] == "linear":
        m, k, n = case["rows"], case["k_dim"], case["n_out"]
        return {"bytes": 2 * (m * k + n * k) + 4 * m * n, "flops": 2 * m * k * n}
    arch, ctx, masks, doms, par = arch_of(case), ints(case["ctx"]), masks_of(case), domains_of(case), parents_of(case)
    d, f, V, L = arch.d_model, arch.d_mlp, arch.vocab, arch.n_layers
    per_layer = 4 * d * d + 3 * d * f
    union = sum(any(not (masks[x] >> l) & 1 for x in doms) for l in range(L))
    if case["kind"] == "grouped":  # one step for every skip set
        union, heads = sum(L - bin(m).count("1") for m in {masks[x] for x in doms}), len({masks[x] for x in doms})
    else:
        heads = 0 if case["kind"] == "prefill" else 1
    rows = sum(len(p) for p in par)
    nbytes, flops = 2 * per_layer * union + heads * 2 * V * d + rows * 2 * d, 0
    for c, p, x in zip(ctx, par, doms):
        act, n = L - bin(masks[x]).count("1"), len(p)
        nbytes += act * (c + n) * 4 * d
        flops += act * (2 * n * per_layer + 4 * d * (n * c + n * (n + 1) // 2))
    if heads:
        nbytes += rows * V * (8 if case["mode"] == "sample" else 4)
        flops += 2 * rows * V * d
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Seen against exact(): the linear layer 2e-6; logits up to 1.4e-4 (activations of 16 bits, fp32
    # sums); cache rows by their rounding to bf16, 1.7e-3 where the whole cache is new (prefill), an
    # ulp (2^-8 of a value) at most.
    if case["kind"] == "linear":
        return {"rel": 1e-5, "max": 1e-4}
    if case["kind"] == "prefill":
        return {"rel": 7e-3, "max": 0.03, "differ": 0.0}
    return {"rel": 2e-3, "max": 0.03, "differ": 0.01}


# ------------------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------------------
def rms(x, g, eps):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * g.double()


def rotate(x, pos, theta):
    """x [n][H][D]: pairs (i, i + D/2) turned by pos * theta^(-2i/D)."""
    half = x.shape[-1] // 2
    inv = theta ** (-torch.arange(half, dtype=torch.float64, device="cuda") * 2 / x.shape[-1])
    a = (pos.double()[:, None] * inv)[:, None, :]
    u, v = x[..., :half], x[..., half:]
    return torch.cat([u * a.cos() - v * a.sin(), v * a.cos() + u * a.sin()], -1)


def exact(case, seed):
    src = Source(seed)
    if case["kind"] == "linear":
        x, w = src.normal(1, (case["rows"], case["k_dim"])), src.normal(2, (case["n_out"], case["k_dim"]), 0.02)
        return x.double() @ w.double().T
    arch, ctx, masks, doms, par = arch_of(case), ints(case["ctx"]), masks_of(case), domains_of(case), parents_of(case)
    H, D, L = arch.n_heads, arch.head_dim, arch.n_layers
    embed, head, gain, nxt = ends(src, arch)
    tok, _ = block_tokens(src, case, arch, nxt)
    h = embed[tok.long()].double()
    rows = [len(p) for p in par]
    at = [sum(rows[:b]) for b in range(len(rows))]
    cap = max(c + n for c, n in zip(ctx, rows)) + 8
    depth, sees = [], []  # per request: row depths and the block rows that a row sees
    for p in par:
        dep = torch.zeros(len(p), dtype=torch.int64)
        see = torch.eye(len(p), dtype=torch.bool)
        for i, q in enumerate(p):
            if q >= 0:
                dep[i] = dep[q] + 1
                see[i] |= see[q]
        depth.append(dep.cuda())
        sees.append(see.cuda())
    kv = []
    for l in range(L):
        reqs = [b for b in range(len(ctx)) if not (masks[doms[b]] >> l) & 1]
        if not reqs:
            continue
        w = layer_weights(src, arch, l)
        cache = torch.zeros((len(ctx), 2, H, cap, D), dtype=torch.float64, device="cuda")
        idx = torch.cat([torch.arange(at[b], at[b] + rows[b], device="cuda") for b in reqs])
        x = rms(h[idx], w["attn_norm"], arch.rms_eps)
        q, k, v = ((x @ w[n].double().T).view(-1, H, D) for n in ("wq", "wk", "wv"))
        out, i0 = torch.empty_like(q), 0
        for b in reqs:
            c, n = ctx[b], rows[b]
            pos = c + depth[b]
            qb = rotate(q[i0:i0 + n], pos, arch.rope_theta)
            kb, vb = rotate(k[i0:i0 + n], pos, arch.rope_theta), v[i0:i0 + n]
            if c:
                cache[b, :, :, :c] = context(src, arch, l, b, c)
            cache[b, 0, :, c:c + n], cache[b, 1, :, c:c + n] = kb.transpose(0, 1), vb.transpose(0, 1)
            # (the cache holds bf16: the block's rows are attended as they are stored)
            ks, vs = (cache[b, j, :, :c + n].to(torch.bfloat16).double() for j in (0, 1))
            s = qb.transpose(0, 1) @ ks.transpose(1, 2) / math.sqrt(D)
            s[:, :, c:].masked_fill_(~sees[b], -math.inf)
            out[i0:i0 + n] = (torch.softmax(s, -1) @ vs).transpose(0, 1)
            i0 += n
        hb = h[idx] + out.reshape(-1, H * D) @ w["wo"].double().T
        x = rms(hb, w["mlp_norm"], arch.rms_eps)
        g = x @ w["w_gate"].double().T
        h[idx] = hb + (g * torch.sigmoid(g) * (x @ w["w_up"].double().T)) @ w["w_down"].double().T
        kv.append(cache)
    if case["kind"] == "prefill":
        return {"kv": kv}
    logits = rms(h, gain, arch.rms_eps) @ head.double().T
    if case["mode"] == "greedy":  # the accepted path's rows follow the context
        best, toks = logits.argmax(-1).tolist(), tok.tolist()
        j = {l: i for i, l in enumerate(l for l in range(L) if any(not (masks[x] >> l) & 1 for x in doms))}
        for b, p in enumerate(par):
            path = [0]
            while True:
                kid = next((i for i, q in enumerate(p) if q == path[-1] and toks[at[b] + i] == best[at[b] + path[-1]]), None)
                if kid is None:
                    break
                path.append(kid)
            for l, i in j.items():
                if not (masks[doms[b]] >> l) & 1:
                    moved = kv[i][b][:, :, [ctx[b] + r for r in path]].clone()
                    kv[i][b][:, :, ctx[b]:ctx[b] + len(path)] = moved
    return {"logits": logits, "accept_len": None, "bonus": None, "path": None, "new_ctx_len": None, "kv": kv}
