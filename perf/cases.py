"""The work a user of this package gives it, as cases that can be timed and compared.

A case is a dict of plain values.  `kind` names the call that a pass makes:

  score    CacheBack.score over one or more senders (strided or paged caches): the part of the
           path that costs most; its scores come back whole
  step     Filter.run: score, select and compact of one sender, outputs included
  chain    Chain.hop three times: each hop's cache is the last hop's message and new positions
  send     Filter.select and Filter.compact on scores that are in hand
  rope     CacheBack.compact_rope: selected rows moved to the receiver's positions
  rows     CacheBack.gather: selected rows of a hidden-state table (the message of embeddings)

Sizes: the workloads of this repository's benchmark and tests (2 to 36 scored layers, 4 to 32
query heads in groups of 1, 2 or 4, head dimension 64 or 128, 64 to 65536 positions, 1 to 640
query tokens) and ragged ones between them.  Inputs follow the same recipe: standard-normal
K, V and Q, and spans of 16 positions whose keys lean towards one query vector.
"""
import math

import torch

import paper_2609_32046_gb300 as cb

SPAN = 16
LATENT = 40
FORCED = 41          # one sink and 40 latent positions


def _case(name, kind, **kw):
    c = dict(kind=kind, layers=36, q_heads=32, kv_heads=8, d=128, senders=1, T=8192, m=64, keep=0.25, p=2.0,
             alpha=2.0, pool=7, page=0, shared=False, self_keys=False)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest state the repository configures (2 layers, d = 64): a call of a few
        # microseconds of device work, where launches and host time count
        _case("tiny_step", "step", layers=2, q_heads=4, kv_heads=2, d=64, T=512, m=16),
        # the benchmark's default: one 8B-shaped sender state of 8192 positions, 64 query tokens
        _case("single_step", "step"),
        # a sequential chain of three agents, each adding 2730 positions to the message it got
        _case("chain_three_hops", "chain", T=2730),
        # fan-in: three agents of 16384 positions scored against one question of 128 tokens
        _case("fanin_score", "score", senders=3, T=16384, m=128),
        # a hybrid model's 8 global-attention layers over a long context
        _case("hybrid_score", "score", layers=8, T=65536),
        # many tasks at once: 24 senders in one call, a query of 64 tokens each
        _case("concurrent_score", "score", senders=24),
        # one state serving eight receivers, whose query tokens also attend to each other
        _case("multiquery_score", "score", senders=8, shared=True, self_keys=True),
        # the cache of a paged server, 16 positions a page, a length that is no multiple of it
        _case("paged_score", "score", T=8191, page=16),
        # a long task description as the query, p and Pool off their defaults
        _case("long_query_score", "score", layers=12, T=6001, m=300, p=3.0, alpha=1.0, pool=5),
        # a model with head dimension 64, ragged length
        _case("d64_score", "score", layers=24, d=64, senders=2, T=7001, m=50),
        # three senders' selected rows gathered into one send buffer
        _case("fanin_send", "send", senders=3, T=16384),
        # the same for one sender, keys turned to the positions they take at the receiver
        _case("reindex", "rope", T=8000),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["score"] * 6 + ["step", "send", "rope", "rows"])
    d = rng.choice([128, 128, 128, 64])
    kv = rng.choice([2, 4, 8, 8])
    G = rng.choice([4, 4, 4, 2, 1])
    while True:
        c = _case(None, kind, layers=_log(rng, 2, 36), q_heads=kv * G, kv_heads=kv, d=d,
                  T=_log(rng, 64, 2048 if kind == "step" else 65536), keep=round(rng.uniform(0.05, 0.6), 3))
        if kind in ("score", "step"):
            c["m"] = _log(rng, 1, 640)
            c["p"] = rng.choice([2.0, 2.0, 2.0, 3.0, 1.5])
            c["alpha"] = rng.choice([2.0, 2.0, 1.0])
            c["pool"] = rng.choice([7, 7, 7, 5, 3, 1])
        if kind in ("score", "send"):
            c["senders"] = rng.choice([1, 1, 1, 2, 3, 5, 8])
        if kind == "score":
            c["page"] = rng.choice([0, 0, 0, 16])
            c["shared"] = c["senders"] > 1 and not c["page"] and rng.random() < 0.3
            c["self_keys"] = rng.random() < 0.2
        logits = c["senders"] * c["layers"] * c["q_heads"] * c["m"] * c["T"]
        nbytes = c["senders"] * c["layers"] * kv * c["T"] * d * 2
        if (kind not in ("score", "step") or logits <= 3e9) and nbytes <= 8e9:
            return c


# --- inputs -----------------------------------------------------------------------------------

def _randn(shape, gen, dtype=torch.bfloat16):
    return torch.randn(shape, generator=gen, device="cuda", dtype=dtype)


def _plant(K, Q, gen, frac=0.05, beta=0.5):
    """5% of the positions, in spans of 16, lean towards one query vector per layer and KV head."""
    nL, Hkv, T, d = K.shape
    m, Hq = Q.shape[1], Q.shape[2]
    G = Hq // Hkv
    spans = max(0, (T - LATENT) // SPAN - 1)
    k = min(spans, max(1, int(frac * T / SPAN)))
    if k < 1:
        return
    at = torch.randperm(spans, generator=gen, device="cuda")[:k] + 1
    pos = (at[:, None] * SPAN + torch.arange(SPAN, device="cuda")).reshape(-1)
    r = torch.randint(0, m, (nL, Hkv), generator=gen, device="cuda")
    h = torch.randint(0, G, (nL, Hkv), generator=gen, device="cuda") + torch.arange(Hkv, device="cuda") * G
    u = Q[torch.arange(nL, device="cuda")[:, None], r, h].float()
    u = beta * u / u.norm(dim=-1, keepdim=True) * math.sqrt(d)
    K[:, :, pos] = (K[:, :, pos].float() + u[:, :, None]).to(K.dtype)


def _inputs(case, seed):
    """K, Q (one per sender or one per pair), the query's own keys."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    nL, Hq, Hkv, d, T, m = (case[k] for k in ("layers", "q_heads", "kv_heads", "d", "T", "m"))
    n = case["senders"]
    Qs = [_randn((nL, m, Hq, d), gen) for _ in range(n)]
    Ks = []
    for i in range(n):
        if case["shared"] and i:
            Ks.append(Ks[0])
            continue
        K = _randn((nL, Hkv, T, d), gen)
        _plant(K, Qs[i], gen)
        Ks.append(K)
    own = [_randn((nL, m, Hkv, d), gen) if case["self_keys"] else None for _ in range(n)]
    return gen, Ks, Qs, own


def _cb(case, m, T, senders):
    return cb.CacheBack(case["layers"], case["q_heads"], case["kv_heads"], case["d"], m, T, senders, p=case["p"],
                        alpha=case["alpha"], pool_width=case["pool"])


def _budget(case):
    return max(cb.budget(case["T"], case["keep"]), min(case["T"], FORCED))


def _paged(K, page, gen):
    """K as the pages of a pool that other sequences share, in a random order."""
    nL, Hkv, T, d = K.shape
    n = -(-T // page)
    total = n + n // 4 + 1
    table = torch.randperm(total, generator=gen, device="cuda")[:n].to(torch.int32)
    pool = torch.zeros((nL, total, page, Hkv, d), dtype=K.dtype, device="cuda")
    full = torch.zeros((nL, n * page, Hkv, d), dtype=K.dtype, device="cuda")
    full[:, :T] = K.permute(0, 2, 1, 3)
    pool[:, table.long()] = full.view(nL, n, page, Hkv, d)
    return cb.PagedKV(pool, pool, table, T)


def _picked(case, gen):
    """Selected positions as the span rule leaves them: whole spans, the sink and the tail."""
    T, B = case["T"], _budget(case)
    score = torch.rand(-(-T // SPAN), generator=gen, device="cuda").repeat_interleave(SPAN)[:T]
    score[:1] = 2
    score[max(0, T - LATENT):] = 2
    return torch.sort(torch.argsort(score, descending=True, stable=True)[:B]).values.to(torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    nL, Hq, Hkv, d, T, m = (case[k] for k in ("layers", "q_heads", "kv_heads", "d", "T", "m"))
    if kind == "score":
        gen, Ks, Qs, own = _inputs(case, seed)
        ctx = _cb(case, m, T, case["senders"])
        out = [torch.empty(T, dtype=torch.float32, device="cuda") for _ in Ks]
        caches = [_paged(K, case["page"], gen) for K in Ks] if case["page"] else Ks
        return dict(kind=kind, ctx=ctx, Ks=caches, Qs=Qs, own=own if case["self_keys"] else None, out=out)
    if kind == "step":
        gen, Ks, Qs, _ = _inputs(case, seed)
        ctx = _cb(case, m, T, 1)
        return dict(kind=kind, filter=cb.Filter(ctx, [(Ks[0], _randn(Ks[0].shape, gen))], Qs, case["keep"]))
    if kind == "chain":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        hops = []
        for _ in range(3):
            Q, K = _randn((nL, m, Hq, d), gen), _randn((nL, Hkv, T, d), gen)
            _plant(K, Q, gen)
            hops.append((Q, K, _randn(K.shape, gen)))
        ctx = _cb(case, m, 3 * T, 1)
        return dict(kind=kind, hops=hops, chain=cb.Chain(ctx, 3 * T, keep=case["keep"], device="cuda"))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = case["senders"]
    ctx = _cb(case, 1, T, n)
    if kind == "rows":
        table = _randn((T, 4096), gen)
        idx = _picked(case, gen)
        return dict(kind=kind, ctx=ctx, table=table, idx=idx,
                    out=torch.empty((len(idx), 4096), dtype=table.dtype, device="cuda"))
    KV = [(_randn((nL, Hkv, T, d), gen), _randn((nL, Hkv, T, d), gen)) for _ in range(n)]
    if kind == "rope":
        idx = _picked(case, gen)
        out = [torch.empty((nL, Hkv, len(idx), d), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        return dict(kind=kind, ctx=ctx, KV=KV[0], idx=idx, out=out)
    # send: positive scores with a heavy tail, neighbours alike, as Pool leaves them
    f = cb.Filter(ctx, KV, [None] * n, case["keep"])
    for s in f.scores:
        base = torch.randn(-(-T // 4), generator=gen, device="cuda").repeat_interleave(4)[:T]
        s.copy_(torch.exp(base + 0.1 * torch.randn(T, generator=gen, device="cuda")) / T)
    return dict(kind=kind, filter=f)


ROPE_BASE = 1e6
ROPE_POS0 = 100


def run(state):
    kind = state["kind"]
    if kind == "score":
        state["ctx"].score(state["Ks"], state["Qs"], state["out"], Kselfs=state["own"])
        return {"scores": state["out"]}
    if kind == "step":
        f = state["filter"].run()
        return {"scores": f.scores, "idx": f.indices(), "k": f.k_out, "v": f.v_out}
    if kind == "chain":
        ch = state["chain"]
        ch.reset()
        hops = [ch.hop(Q, K, V) for Q, K, V in state["hops"]]
        return {"scores": [h["scores"] for h in hops], "idx": [h["idx"] for h in hops],
                "k": hops[-1]["message_K"], "v": hops[-1]["message_V"]}
    if kind == "send":
        f = state["filter"]
        f.select()
        f.compact()
        return {"idx": f.indices(), "k": f.k_out, "v": f.v_out}
    if kind == "rope":
        K, V = state["KV"]
        idx, (k, v) = state["idx"], state["out"]
        state["ctx"].compact_rope([K], [V], [idx], [len(idx)], k, v, [0], ROPE_BASE, pos0=ROPE_POS0)
        return {"k": k, "v": v}
    state["ctx"].gather([state["table"]], [state["idx"]], [len(state["idx"])], state["out"], [0])
    return {"rows": state["out"]}


# --- what a pass cannot do without --------------------------------------------------------------

def work(case):
    nL, Hq, Hkv, d, T, m, n = (case[k] for k in ("layers", "q_heads", "kv_heads", "d", "T", "m", "senders"))
    B = _budget(case)
    row = nL * Hkv * d * 2                       # bytes of one position's K (or V)

    def score(T, pairs, states):
        return {"bytes": states * T * row + pairs * (nL * m * Hq * d * 2 + 4 * T), "flops": 2 * pairs * nL * m * Hq * T * d}

    kind = case["kind"]
    if kind == "score":
        return score(T, n, 1 if case["shared"] else n)
    if kind == "step":
        w = score(T, 1, 1)
        return {"bytes": w["bytes"] + 4 * B * row + 4 * B, "flops": w["flops"]}
    if kind == "chain":
        total, old = {"bytes": 0, "flops": 0}, 0
        for _ in range(3):
            w = score(old + T, 1, 1)
            B = max(cb.chain_budget(old, T, case["keep"]), min(old + T, FORCED))
            # the new rows into the chain's buffer, the kept rows into the next one
            total["bytes"] += w["bytes"] + 4 * T * row + 4 * B * row
            total["flops"] += w["flops"]
            old = B
        return total
    if kind == "send":
        return {"bytes": n * (4 * T + 4 * B + 4 * B * row), "flops": 0}
    if kind == "rope":
        return {"bytes": 4 * B * row + 4 * B, "flops": 0}
    return {"bytes": 2 * B * 4096 * 2 + 4 * B, "flops": 0}


def tolerance(case):
    kind = case["kind"]
    if kind in ("send", "rows"):
        return "exact"                           # indices and copied bytes
    if kind == "rope":
        # one rounding to bf16 of each rotated value (2^-9 of it at most); another correct angle
        # reduction flips a few of these roundings
        return {"rel": 5e-3, "max": 2e-2}
    # scores: 32-bit sums over layers, heads and query tokens of exponentials of 32-bit logits;
    # whole calls also return the rows that the scores select, where a tie may fall either way
    tol = {"rel": 1e-5, "max": 1e-4}
    if kind in ("step", "chain"):
        tol["differ"] = 0.01
    return tol


# --- the same in 64 bits --------------------------------------------------------------------------

def _pool(x, w):
    if w == 1:
        return x
    y = torch.nn.functional.pad(x, (w // 2, w // 2), value=0.0)
    T = x.shape[-1]
    out = y[..., :T]
    for k in range(1, w):
        out = torch.maximum(out, y[..., k:k + T])
    return out


def _exact_scores(case, K, Q, own):
    """Scores of one sender in 64 bits: softmax over positions (and the query tokens' own keys up
    to each token), head means b, Q = Pool(mean), C = (sum Pool(b)^p / sum Pool(mean b)^p)^(1/(p-1))."""
    nL, Hkv, T, d = K.shape
    m, Hq = Q.shape[1], Q.shape[2]
    G, p, w = Hq // Hkv, case["p"], case["pool"]
    U = torch.zeros(T, dtype=torch.float64, device=K.device)
    N, D = torch.zeros_like(U), torch.zeros_like(U)
    for l in range(nL):
        for g in range(Hkv):
            q = Q[l, :, g * G:(g + 1) * G].double()                       # [m][G][d]
            z = (q.reshape(m * G, d) @ K[l, g].double().T).view(m, G, T) / math.sqrt(d)
            if own is not None:
                zs = (q.reshape(m * G, d) @ own[l, :, g].double().T).view(m, G, m) / math.sqrt(d)
                later = torch.ones(m, m, dtype=torch.bool, device=K.device).triu(1)
                zs = zs.masked_fill(later[:, None, :], -math.inf)
                a = torch.softmax(torch.cat([z, zs], -1), -1)[..., :T]
            else:
                a = torch.softmax(z, -1)
            b = a.mean(1)
            mean = b.mean(0)
            U += mean / Hkv
            N += _pool(b, w).pow_(p).mean(0)
            D += _pool(mean, w) ** p
    C = torch.where(D > 0, (N / D) ** (1.0 / (p - 1.0)), torch.ones_like(D))
    return _pool(U, w) * C ** case["alpha"]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("score", "step"):
        _, Ks, Qs, own = _inputs(case, seed)
        s = [_exact_scores(case, K, Q, o) for K, Q, o in zip(Ks, Qs, own)]
        if kind == "score":
            return {"scores": s}
        return {"scores": s, "idx": None, "k": None, "v": None}
    if kind == "chain":
        # the first hop's scores; the later hops' caches depend on what the first selects
        st = prepare(case, seed)
        Q, K, _ = st["hops"][0]
        return {"scores": [_exact_scores(case, K, Q, None), None, None], "idx": None, "k": None, "v": None}
    if kind == "rope":
        st = prepare(case, seed)
        K, V = st["KV"]
        idx = st["idx"].long()
        d = case["d"]
        k = K[:, :, idx].double()
        turn = (ROPE_POS0 + torch.arange(len(idx), device=K.device) - idx).double()
        a = turn[:, None] * ROPE_BASE ** (-torch.arange(0, d, 2, device=K.device).double() / d)
        x, y = k[..., : d // 2], k[..., d // 2:]
        out = torch.cat([x * a.cos() - y * a.sin(), y * a.cos() + x * a.sin()], -1)
        return {"k": out, "v": V[:, :, idx].double()}
    return None
