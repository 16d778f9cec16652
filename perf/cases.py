"""Performance cases of the draft-and-verify path: what a decoding program asks of the library, through its public calls.

Kinds: `attn` (tree attention of one verification pass), `accept` (greedy acceptance from logits), `draft` (table update and
draft tree of one step), `ingest` (prompt into the tables, then the first draft), `frozen` (the read-only table built from a
corpus, then drafted from) and `step` (one whole decoding step at small batch, captured in a CUDA graph as a serving loop
captures it).  Shapes are those of the workload configurations; contexts and tree sizes are spread evenly over the stated range
and dealt to the sequences by the seed, so that the work of a case does not depend on it.
"""
import math

import numpy as np
import torch

from paper_2511_21699_b200 import api

DEV = "cuda:0"
PAGE = 16


# ---------------------------------------------------------------------------------------------------- the cases
def _attn(name, batch, hq, hkv, d, lo, hi, t, trees):
    return dict(name=name, kind="attn", batch=batch, hq=hq, hkv=hkv, d=d, ctx_lo=lo, ctx_hi=hi, t=t, trees=trees)


def _accept(name, batch, t, vocab, dtype, trees):
    return dict(name=name, kind="accept", batch=batch, t=t, vocab=vocab, dtype=dtype, trees=trees)


def _draft(name, batch, ll, fl, lc, fc, t, depth, crt, hist, new, vocab):
    return dict(name=name, kind="draft", batch=batch, ll=ll, fl=fl, lc=lc, fc=fc, t=t, depth=depth, crt=crt, hist=hist, new=new, vocab=vocab)


def _ingest(name, batch, ll, fl, lc, fc, lo, hi, vocab, scratch):
    return dict(name=name, kind="ingest", batch=batch, ll=ll, fl=fl, lc=lc, fc=fc, ctx_lo=lo, ctx_hi=hi, vocab=vocab, scratch=scratch, t=64, depth=8, crt=16)


def _frozen(name, tokens, ll, fl, lc, fc, vocab):
    return dict(name=name, kind="frozen", tokens=tokens, ll=ll, fl=fl, lc=lc, fc=fc, vocab=vocab, batch=32, t=64, depth=8, crt=16)


def _step(name, batch, hq, hkv, d, ctx, t, ll, fl, lc, fc, depth, crt, vocab):
    return dict(name=name, kind="step", batch=batch, hq=hq, hkv=hkv, d=d, ctx_lo=ctx, ctx_hi=ctx, t=t, ll=ll, fl=fl, lc=lc, fc=fc, depth=depth,
                crt=crt, vocab=vocab, trees="full")


def listed():
    return [
        # one user's chat on a 7B-shaped model: a single sequence, every layer calls this once per step
        _attn("attn_b1_4k_mha", 1, 32, 32, 128, 4096, 4096, 64, "full"),
        # a server's batch of ragged contexts on an 8B-shaped model with grouped heads
        _attn("attn_b32_ragged_gqa4", 32, 32, 8, 128, 1024, 8192, 64, "full"),
        # multi-turn chats on a 13B-shaped model without grouped heads: many short units
        _attn("attn_b64_2k_mha", 64, 40, 40, 128, 2048, 2048, 32, "full"),
        # long contexts, large trees and a large batch on a 70B-shaped model: the largest call
        _attn("attn_b128_32k_gqa8", 128, 64, 8, 128, 32768, 32768, 128, "full"),
        # the same server with the drafter's own small and uneven trees, head_dim 64 and contexts that are no round numbers
        _attn("attn_b13_odd_d64_small_trees", 13, 32, 8, 64, 777, 5003, 61, "ragged"),
        # acceptance of a server's batch over a 128 k vocabulary, fp32 logits
        _accept("accept_b32_v128k_f32", 32, 64, 128256, "f32", "full"),
        # acceptance of one sequence, bf16 logits as a serving model's head emits them
        _accept("accept_b1_v32k_bf16", 1, 64, 32000, "bf16", "full"),
        # the drafter of the large batch: five new tokens per sequence go into the tables, then 128 trees are grown
        _draft("draft_b128_64k_leaders", 128, 3, 5, 65536, 8, 128, 10, 32, 8192, 5, 128256),
        # the paper's tuned table (unigram leaders, 128 followers each) for one sequence
        _draft("draft_b1_tuned", 1, 1, 3, 1 << 20, 128, 96, 24, 16, 4097, 3, 32000),
        # prompts of a server's batch go into empty tables
        _ingest("ingest_b32_ragged", 32, 3, 4, 16384, 4, 1024, 8192, 128256, True),
        # the read-only table built from a corpus sample
        _frozen("frozen_4m_bigram", 4 << 20, 2, 4, 65536, 8, 32000),
        # a whole step of one user's chat as a graph: verification attention, acceptance with the next draft, key/value commit
        _step("step_b1_7b", 1, 32, 32, 128, 4096, 64, 2, 4, 16384, 4, 8, 16, 32000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["attn", "attn", "attn", "accept", "draft", "draft", "ingest", "frozen", "step"])
    if kind == "attn":
        hq, hkv = rng.choice([(8, 8), (32, 32), (40, 40), (32, 8), (64, 8), (16, 4)])
        d = rng.choice([64, 128, 128])
        t = _log_int(rng, 3, 128)
        batch = _log_int(rng, 1, 128)
        room = min(16384, int(4e9 / (batch * hkv * d * 4)), int(2e12 / (4.0 * hq * d * t * batch)))
        hi = _log_int(rng, 65, max(66, room))
        lo = hi if rng.random() < 0.3 else max(1, int(hi * rng.uniform(0.1, 0.9)))
        c = _attn("", batch, hq, hkv, d, lo, hi, t, rng.choice(["full", "full", "ragged"]))
    elif kind == "accept":
        vocab = rng.choice([32000, 128256, 151936, 50257])
        batch = _log_int(rng, 1, 96)
        t = _log_int(rng, 2, 128)
        while batch * t * vocab * 4 > 2e9:
            batch = max(1, batch // 2)
            t = t if batch > 1 else t // 2
        c = _accept("", batch, t, vocab, rng.choice(["f32", "bf16"]), rng.choice(["full", "ragged"]))
    elif kind == "draft":
        ll = rng.choice([1, 2, 2, 3])
        fc = rng.choice([4, 6, 8, 32, 40, 128]) if ll == 1 else rng.choice([4, 4, 6, 8])
        t = _log_int(rng, 16, 128)
        c = _draft("", _log_int(rng, 1, 128), ll, rng.choice([3, 4, 5]), rng.choice([8192, 16384, 65536]), fc, t, rng.choice([6, 8, 10, 24]), t // 4,
                   _log_int(rng, 600, 7600), rng.randint(1, 8), rng.choice([32000, 128256]))
    elif kind == "ingest":
        hi = _log_int(rng, 300, 8000)
        c = _ingest("", _log_int(rng, 1, 96), rng.choice([1, 2, 3]), rng.choice([3, 4, 5]), rng.choice([8192, 16384]), rng.choice([4, 6, 8]),
                    max(20, int(hi * rng.uniform(0.2, 1.0))), hi, rng.choice([32000, 128256]), rng.random() < 0.75)
    elif kind == "frozen":
        ll = rng.choice([1, 2, 3])
        c = _frozen("", _log_int(rng, 60001, 4 << 20), ll, rng.choice([3, 4]), rng.choice([16384, 65536]), rng.choice([8, 16, 64]), 32000)
    else:
        hq, hkv = rng.choice([(32, 32), (32, 8), (8, 8)])
        t = _log_int(rng, 16, 96)
        c = _step("", rng.randint(1, 6), hq, hkv, rng.choice([64, 128]), _log_int(rng, 200, 7000), t, rng.choice([1, 2]), rng.choice([3, 4]), 16384,
                  rng.choice([4, 8]), 8, t // 4, 32000)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------------- inputs
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 64 + salt)
    return g


def _spread(lo, hi, n):
    """n whole numbers spread evenly over [lo, hi]; the largest is hi."""
    return np.array([hi], np.int64) if n == 1 else np.round(np.linspace(lo, hi, n)).astype(np.int64)


def _ctx(case, seed):
    c = _spread(case["ctx_lo"], case["ctx_hi"], case["batch"])
    return np.random.RandomState(seed).permutation(c).astype(np.int32)


def _nodes(case, seed):
    B, T = case["batch"], case["t"]
    n = np.full(B, T, np.int64) if case["trees"] == "full" else (_spread(1, T, B) if B > 1 else np.array([max(1, T // 3)]))
    return np.random.RandomState(seed + 1).permutation(n).astype(np.int32)


def _streams(seed, batch, length, vocab, copy=0.35, span=(4, 32), s=1.08):
    """int32 [batch, length]: Zipf-distributed ids with stretches that repeat earlier text."""
    g = _gen(seed, 1)
    cdf = torch.cumsum(torch.arange(1, vocab + 1, device=DEV, dtype=torch.float64) ** -s, 0)
    u = torch.rand(batch, length, generator=g, device=DEV, dtype=torch.float64) * cdf[-1]
    rank = torch.searchsorted(cdf, u).clamp_(max=vocab - 1)
    a = 2654435761 % vocab
    while math.gcd(a, vocab) != 1:
        a += 1
    ids = (rank * a + 12345) % vocab
    mean = 0.5 * (span[0] + span[1])
    pieces = 2 * (int(length * copy / mean) * 2 + 8)
    gaps = (-torch.log(torch.rand(batch, pieces // 2, generator=g, device=DEV).clamp_(min=1e-7)) * mean * (1 - copy) / copy).long() + 1
    spans = torch.randint(span[0], span[1] + 1, (batch, pieces // 2), generator=g, device=DEV)
    starts = torch.cumsum(torch.stack([gaps, spans], 2).reshape(batch, pieces), 1)
    starts = torch.cat([torch.zeros(batch, 1, dtype=torch.long, device=DEV), starts[:, :-1]], 1)     # piece 2k: a gap, 2k + 1: a span
    pos = torch.arange(length, device=DEV).expand(batch, length).contiguous()
    piece = torch.searchsorted(starts, pos, right=True) - 1
    begin = starts.gather(1, piece)
    src = (torch.rand(batch, pieces, generator=g, device=DEV).gather(1, piece) * begin).long() + pos - begin
    at = torch.where((piece % 2 == 1) & (begin > 0), src, pos)
    for _ in range(20):
        at = at.gather(1, at)
    return ids.gather(1, at).to(torch.int32).contiguous()


def _trees(case, seed, max_depth):
    """Random trees, parents before children: dict of device arrays as the drafter writes them (token = 1 + node number, times 7)."""
    B, T = case["batch"], case["t"]
    r = np.random.RandomState(seed + 2)
    n = _nodes(case, seed)
    par = np.full((B, T), -1, np.int64)
    dep = np.full((B, T), -1, np.int64)
    dep[:, 0] = 0
    W = (T + 31) // 32
    mask = np.zeros((B, T, W), np.uint32)
    mask[:, 0, 0] = 1
    rows = np.arange(B)
    for i in range(1, T):
        p = np.where(r.rand(B) < 0.5, r.randint(0, i, B), i - 1)
        p = np.where(dep[rows, p] < max_depth, p, 0)
        par[:, i] = p
        dep[:, i] = dep[rows, p] + 1
        mask[:, i] = mask[rows, p]
        mask[:, i, i // 32] |= np.uint32(1) << np.uint32(i % 32)
    tok = np.tile((np.arange(T) + 1) * 7, (B, 1))
    gone = np.arange(T)[None, :] >= n[:, None]
    for a in (par, dep, tok):
        a[gone] = -1
    mask[gone] = 0
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x.astype(np.int32))).to(DEV)  # noqa: E731
    return dict(tokens=d(tok), parent=d(par), depth=d(dep), mask=torch.from_numpy(mask.view(np.int32)).to(DEV), n_nodes=d(n))


def _attn_inputs(case, seed, extra_tokens=0):
    B, T, hq, hkv, D = (case[k] for k in ("batch", "t", "hq", "hkv", "d"))
    ctx = _ctx(case, seed)
    pages = (ctx.astype(np.int64) + extra_tokens + PAGE - 1) // PAGE
    total = int(pages.sum()) + 3
    g = _gen(seed, 2)
    bf = dict(dtype=torch.bfloat16, device=DEV)
    normal = lambda *shape: torch.empty(*shape, **bf).normal_(generator=g)  # noqa: E731
    perm = np.random.RandomState(seed + 3).permutation(total).astype(np.int32)
    table = np.full((B, int(pages.max())), -1, np.int32)
    at = 0
    for b in range(B):
        table[b, : pages[b]] = perm[at:at + pages[b]]
        at += int(pages[b])
    return dict(q=normal(B, T, hq, D), k_pool=normal(total, PAGE, hkv, D), v_pool=normal(total, PAGE, hkv, D),
                block_table=torch.from_numpy(table).to(DEV), ctx_len=torch.from_numpy(ctx).to(DEV), k_tree=normal(B, T, hkv, D),
                v_tree=normal(B, T, hkv, D))


def _logits(case, seed, tree):
    """[B, T, V] with the token of some child of most nodes planted as the row's maximum."""
    B, T, V = case["batch"], case["t"], case["vocab"]
    x = torch.empty(B, T, V, dtype=torch.float32 if case.get("dtype", "f32") == "f32" else torch.bfloat16, device=DEV).normal_(generator=_gen(seed, 3))
    par, tok = tree["parent"].long(), tree["tokens"].long()
    keep = (par >= 0) & (torch.rand(B, T, generator=_gen(seed, 4), device=DEV) < 0.6)
    b = torch.arange(B, device=DEV)[:, None].expand(B, T)
    x[b[keep], par[keep], tok[keep] % V] = 32.0
    return x


def _context(case, max_nodes=None, heads=(8, 8, 64)):
    hq, hkv, d = (case["hq"], case["hkv"], case["d"]) if "hq" in case else heads
    return api.Cacheback(case["batch"], case.get("ll", 2), case.get("fl", 4), case.get("lc", 64), case.get("fc", 4), max_nodes or case["t"],
                         case.get("crt", 0), case.get("depth", 10), case.get("vocab", 32000), hq, hkv, d, PAGE, 0, DEV)


def _i32(x):
    return torch.from_numpy(np.ascontiguousarray(x).astype(np.int32)).to(DEV)


def prepare(case, seed):
    kind, B = case["kind"], case["batch"]
    s = dict(kind=kind)
    if kind == "attn":
        s.update(_attn_inputs(case, seed), tree=_trees(case, seed, 10), cb=_context(case), max_ctx=case["ctx_hi"])
        s["out"] = torch.empty_like(s["q"])
        s["lse"] = torch.empty(B, case["hq"], case["t"], dtype=torch.float32, device=DEV)
    elif kind == "accept":
        s.update(tree=_trees(case, seed, 10), cb=_context(case))
        s["logits"] = _logits(case, seed, s["tree"])
        s["res"] = s["cb"].alloc_accept()
    elif kind == "draft":
        hist, new = case["hist"], case["new"]
        s.update(tokens=_streams(seed, B, hist + new, case["vocab"]), cb=_context(case), n_old=_i32(np.full(B, hist)), n_new=_i32(np.full(B, hist + new)))
        s["cb"].cb_bulk_scratch_attach(B * hist)
        s["cb"].cb_update_bulk(s["tokens"], _i32(np.zeros(B)), s["n_old"])
        torch.cuda.synchronize()
        s["cb"].cb_bulk_scratch_attach(None)
        s["tree"] = s["cb"].alloc_tree()
    elif kind == "ingest":
        n = _ctx(case, seed)
        s.update(tokens=_streams(seed, B, int(n.max()), case["vocab"]), cb=_context(case), zero=_i32(np.zeros(B)), n=_i32(n))
        if case["scratch"]:
            s["cb"].cb_bulk_scratch_attach(int(n.sum()))
        s["tree"] = s["cb"].alloc_tree()
    elif kind == "frozen":
        corpus = _streams(seed, 1, case["tokens"], case["vocab"])[0].contiguous()
        step = max(1, (case["tokens"] - 64) // B)
        tokens = torch.stack([corpus[k * step:k * step + 64] for k in range(B)]).contiguous()
        s.update(corpus=corpus, tokens=tokens, n=_i32(np.full(B, 64)), cb=_context(case), table=api.FrozenTable(case["ll"], case["fl"], case["lc"], case["fc"], DEV))
        s["tree"] = s["cb"].alloc_tree()
    else:
        s.update(_attn_inputs(case, seed, extra_tokens=64), cb=_context(case))
        hist = case["ctx_hi"] + 1
        tokens = _streams(seed, B, hist + 64, case["vocab"])
        n = _i32(np.full(B, hist))
        cb = s["cb"]
        cb.cb_update_bulk(tokens, _i32(np.zeros(B)), n)
        tree = _trees(case, seed, case["depth"])
        logits = _logits(case, seed, tree)
        nxt, res = cb.alloc_tree(), cb.alloc_accept()
        out = torch.empty_like(s["q"])
        length, ctx = n.clone(), s["ctx_len"].clone()

        def step():
            length.copy_(n)
            ctx.copy_(s["ctx_len"])
            cb.cb_tree_attn(s["q"], s["k_pool"], s["v_pool"], s["block_table"], ctx, s["k_tree"], s["v_tree"], tree["mask"], tree["n_nodes"], out=out,
                            max_ctx=case["ctx_hi"])
            cb.cb_accept_update_draft_tree(tree, logits, tokens, length, next_tree=nxt, res=res)
            cb.cb_kv_commit(s["k_pool"], s["v_pool"], s["block_table"], ctx, s["k_tree"], s["v_tree"], res["n_accept"], res["accept_nodes"])

        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            step()
        torch.cuda.current_stream().wait_stream(side)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            step()
        s.update(graph=graph, hold=(tree, logits, tokens, n), answer=dict(out=out, next=nxt, res=res, length=length, ctx=ctx))
    return s


def run(s):
    kind, cb = s["kind"], s["cb"]
    if kind == "attn":
        cb.cb_tree_attn(s["q"], s["k_pool"], s["v_pool"], s["block_table"], s["ctx_len"], s["k_tree"], s["v_tree"], s["tree"]["mask"],
                        s["tree"]["n_nodes"], out=s["out"], lse=s["lse"], max_ctx=s["max_ctx"])
        return dict(out=s["out"], lse=s["lse"])
    if kind == "accept":
        return cb.cb_accept(s["tree"], logits=s["logits"], res=s["res"])
    if kind == "draft":
        return cb.cb_update_draft_tree(s["tokens"], s["n_old"], s["n_new"], s["tree"])
    if kind == "ingest":
        cb.cb_reset()
        cb.cb_update_bulk(s["tokens"], s["zero"], s["n"])
        return cb.cb_draft_tree(s["tokens"], s["n"], s["tree"])
    if kind == "frozen":
        s["table"].cb_frozen_build(s["corpus"])
        cb.cb_frozen_attach(s["table"])
        return cb.cb_draft_tree(s["tokens"], s["n"], s["tree"])
    s["graph"].replay()
    return s["answer"]


# ---------------------------------------------------------------------------------------------------- work, tolerance, exact
def work(case):
    kind, B, T = case["kind"], case["batch"], case["t"]
    entry = 4 * (case.get("ll", 0) + case.get("fc", 0) * (1 + case.get("fl", 0)))
    tree_out = B * T * (12 + 4 * ((T + 31) // 32))
    bytes_, flops = 0.0, 0.0
    if kind in ("attn", "step"):
        ctx, n = _ctx(case, 0).astype(np.int64), _nodes(case, 0).astype(np.int64)
        # keys and values of two independent permutations: contexts and tree sizes are dealt out separately
        mean_n = float(n.mean())
        bytes_ += float(ctx.sum()) * case["hkv"] * case["d"] * 4 + float(n.sum()) * case["d"] * 4 * (case["hkv"] + case["hq"])
        flops += 4.0 * case["hq"] * case["d"] * float(ctx.sum()) * mean_n
    if kind == "accept":
        bytes_ += float(_nodes(case, 0).sum()) * case["vocab"] * (4 if case["dtype"] == "f32" else 2) + B * T * 16
    if kind == "step":
        bytes_ += float(B) * T * case["vocab"] * 4
    if kind in ("draft", "step"):
        # per new token a window: its bucket and entry read and written; per tree at least the root's lookup
        bytes_ += B * (case.get("new", 4) * 2 + 1) * (128 + entry) + tree_out
    if kind == "ingest":
        windows = float(_ctx(case, 0).sum())
        bytes_ += windows * 4 + windows * 0.7 * entry + B * (128 + entry) + tree_out
    if kind == "frozen":
        bytes_ += case["tokens"] * 4.0 + case["lc"] * entry + tree_out
    return dict(bytes=bytes_, flops=flops)


def tolerance(case):
    # integers everywhere but in attention, whose probabilities are rounded to bf16 before the product with the values and
    # whose output is bf16
    return {"rel": 1e-2, "max": 5e-2} if case["kind"] in ("attn", "step") else "exact"


def exact(case, seed):
    if case["kind"] not in ("attn", "step"):
        return None
    x = _attn_inputs(case, seed, extra_tokens=64 if case["kind"] == "step" else 0)
    tree = _trees(case, seed, 10 if case["kind"] == "attn" else case["depth"])
    B, T, hq, hkv, D = (case[k] for k in ("batch", "t", "hq", "hkv", "d"))
    G = hq // hkv
    out = torch.zeros(B, T, hq, D, dtype=torch.float64, device=DEV)
    lse = torch.zeros(B, hq, T, dtype=torch.float64, device=DEV)
    ctx, nodes = x["ctx_len"].tolist(), tree["n_nodes"].tolist()
    word = torch.arange(T, device=DEV) // 32
    bit = torch.arange(T, device=DEV) % 32
    for b in range(B):
        c, n = ctx[b], nodes[b]
        pages = x["block_table"][b, : (c + PAGE - 1) // PAGE].long()
        sees = ((tree["mask"][b][:, word] >> bit) & 1).bool()[:n, :n]                        # [n, n]: node i sees node j
        for h in range(hkv):
            k = torch.cat([x["k_pool"][pages, :, h].reshape(-1, D)[:c], x["k_tree"][b, :n, h]]).double()
            v = torch.cat([x["v_pool"][pages, :, h].reshape(-1, D)[:c], x["v_tree"][b, :n, h]]).double()
            q = x["q"][b, :n, h * G:(h + 1) * G].double().permute(1, 0, 2).reshape(G * n, D)
            sc = (q @ k.T).view(G, n, c + n) / math.sqrt(D)
            sc[:, :, c:].masked_fill_(~sees, -math.inf)
            l = torch.logsumexp(sc, -1)
            out[b, :n, h * G:(h + 1) * G] = (torch.exp(sc - l[..., None]).view(G * n, c + n) @ v).view(G, n, D).permute(1, 0, 2)
            lse[b, h * G:(h + 1) * G, :n] = l
    return dict(out=out, lse=lse) if case["kind"] == "attn" else dict(out=out)
