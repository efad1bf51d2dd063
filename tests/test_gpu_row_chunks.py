"""The tcgen05 score passes over head dimension 64, many query rows and the edges of their tiles.

Pass 1 takes 128-position tiles and up to 512 query rows at a time, pass 2 blocks of 480 output
positions (four tiles of every fourth position, the last T mod 4 positions read through a map of
their own) or of 104, and up to 256 rows at a time; rows come in halves of 128.

Tolerance: a logit is a 32-bit sum of at most 128 products of bf16 values, off by less than
128 * 2^-24 * sum |q k| / sqrt(d) < 1e-4 and by about its square root's share, 1e-6, in practice;
the row's offset adds 2^-24 of itself.  A score is a mean of exponentials times the square of a
ratio of such means, so its relative error is a few times the logits': 5e-5 bounds it.
"""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_2609_32046_gb300 as cb
import synth
from gpu_helpers import assert_scores_close, check_sender, make_cb, oracle_scores, run_path

pytestmark = pytest.mark.gpu

RTOL = 5e-5

# (nL, Hq, Hkv, d), T list, m, extra config
CASES = [
    ((2, 4, 2, 64), [512], 80, {}),
    ((1, 8, 4, 64), [481], 257, {}),                    # 514 rows: five halves in two row chunks (pass 1), three (pass 2)
    ((1, 2, 2, 64), [1025], 300, dict(p=3.0, pool_width=5)),
    ((2, 16, 4, 64), [700, 77, 4], 128, {}),            # 512 rows: one row chunk of pass 1, two of pass 2
    ((1, 16, 4, 128), [961], 129, {}),                  # 516 rows
    ((1, 8, 2, 128), [479], 300, {}),                   # 1200 rows
    ((1, 4, 2, 128), [130], 700, dict(p=1.5)),          # 1400 rows, G = 2
    ((1, 2, 2, 128), [77], 1024, {}),                   # the most query tokens
    ((1, 8, 2, 128), [600], 150, dict(p=float("inf"))),  # maxima over row chunks
    ((1, 8, 2, 64), [333], 65, dict(self_keys=True)),
    ((1, 8, 2, 64), [300], 130, dict(self_keys=True)),  # the self keys fill a tile and part of a second
    # last chunks of one and six positions: most column quarters of a tile see self keys alone
    ((1, 8, 2, 128), [1030, 1025, 5, 129], 100, dict(self_keys=True)),
    ((1, 8, 2, 128), [1, 2, 3, 5, 119, 120, 121, 122, 480, 481, 482, 483], 5, {}),
    ((1, 8, 2, 64), [1, 3, 121, 479, 480, 483], 66, dict(pool_width=1)),
    # fewer blocks than SMs
    ((1, 2, 2, 128), [1000], 20, dict(pool_width=1, p=3.0)),
    ((2, 16, 4, 128), [2106], 24, dict(p=3.0)),
    ((8, 8, 4, 128), [2400], 24, dict(pool_width=1, p=float("inf"))),
]


@pytest.mark.parametrize("case", CASES, ids=["d%d_g%d_m%d_T%d" % (c[0][3], c[0][1] // c[0][2], c[2], c[1][0])
                                             for c in CASES])
def test_scores(case):
    shape, Ts, m, extra = case
    extra = dict(extra)
    w = synth.custom_workload(synth.Shape(*shape), Ts, m, seed=m + Ts[0], n_planted_spans=2)
    qk = [synth.make_query_keys(w.spec, 5, s.task) for s in w.senders] if extra.pop("self_keys", False) else None
    f = run_path(w, 0.3, query_keys=qk, **extra)
    assert f.cb.score_path() == 2
    o = oracle.default()
    for i, s in enumerate(w.senders):
        kself = None if qk is None else qk[i]
        ref = oracle_scores(o, s.K, w.queries[s.task], p=extra.get("p", 2.0), pool_w=extra.get("pool_width", 7),
                            Kself=kself)
        assert_scores_close(f.scores[i].cpu().numpy(), ref["S"], rtol=RTOL)
        check_sender(f, i, s.K, s.V, w.queries[s.task], p=extra.get("p", 2.0), pool_w=extra.get("pool_width", 7),
                     Kself=kself)


def _attention_64(K, Q, Ts):
    """b[group, token, position] in 64 bits (softmax over positions, mean over a group's heads), per T."""
    nL, Hkv, _, d = K.shape
    m, G = Q.shape[1], Q.shape[2] // Hkv
    q = Q.double().view(nL, m, Hkv, G, d).permute(0, 2, 1, 3, 4).reshape(nL, Hkv, m * G, d)
    z = q @ K.double().transpose(-1, -2) / math.sqrt(d)
    return [torch.softmax(z[..., :T], -1).view(nL * Hkv, m, G, T).mean(2) for T in Ts]


def _score_64(b, Hkv, width, p):
    """Scores (alpha = 2) of b by their definition."""
    widest = lambda x: torch.nn.functional.max_pool1d(x, width, 1, width // 2)
    U, N, D = widest(b.sum(0).mean(0)[None])[0] / Hkv, widest(b), widest(b.mean(1))
    if math.isinf(p):
        return U * (N.amax((0, 1)) / D.amax(0)) ** 2
    return U * ((N ** p).mean(1).sum(0) / (D ** p).sum(0)) ** (2 / (p - 1))


@pytest.mark.parametrize("few", [False, True], ids=["full", "few"])
@pytest.mark.parametrize("G", [1, 2, 4])
@pytest.mark.parametrize("d", [64, 128])
def test_every_pass_2_instantiation(d, G, few):
    """k_accum_tc<d, G, pool_width / 2, p = 2, another or infinity, few>: `few` where a sender's last 128
    query rows are at most 64.  26 groups, so that three blocks of 480 positions are more than the units
    that go by blocks of one tile; T around the ends of blocks and lane quarters, each remainder of four."""
    m = {1: 140, 2: 66, 4: 66}[G] if few else {1: 100, 2: 100, 4: 90}[G]
    nL, Hkv, Ts = 13, 2, [1440, 1441, 1442, 1443, 1559, 1560, 1561, 1700]
    gen = torch.Generator(device="cuda").manual_seed(10 * d + G)
    draw = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    K, Q = draw(nL, Hkv, max(Ts), d), draw(nL, m, Hkv * G, d)
    bs, out = _attention_64(K, Q, Ts), [torch.empty(T, device="cuda") for T in Ts]
    for width in (1, 3, 5, 7):
        for p in (2.0, 3.0, float("inf")):
            c = cb.CacheBack(nL, Hkv * G, Hkv, d, m, max(Ts), len(Ts), p=p, pool_width=width)
            c.score([K[:, :, :T] for T in Ts], [Q] * len(Ts), out)
            c.sync_status()
            assert c.score_path() == 2
            for b, got in zip(bs, out):
                assert_scores_close(got.cpu().numpy(), _score_64(b, Hkv, width, p).cpu().numpy(), rtol=RTOL)


@pytest.mark.parametrize("G,width,p", [(1, 7, 2.0), (1, 1, 3.0), (2, 5, 2.0), (2, 3, float("inf")), (4, 7, 3.0),
                                       (4, 5, float("inf")), (4, 1, 2.0), (2, 7, 2.0), (1, 3, 1.5)])
@pytest.mark.parametrize("d", [64, 128])
def test_few_rows_and_short_senders(d, G, width, p):
    """Pass 2 hands a half's columns to the warps in eights up to 64 rows, and takes senders of up to 312
    positions (d = 64: 208), or of up to 33 blocks of 480, in blocks of one tile (104 outputs): both
    sides of each line, in one call; every sender's scores are also those of a call of its own."""
    nL, Hkv, Ts = 9, 4, [1, 26, 104, 105, 208, 209, 312, 313, 1100]   # 36 groups
    gen = torch.Generator(device="cuda").manual_seed(d + G)
    draw = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    for rows in (4, 32, 36, 64, 68, 96, 100, 128, 132, 196, 264, 516):
        m = rows // G
        if d == 64 and m <= 64:
            m += 64          # (fewer tokens: the mma.sync passes)
        K, Q = draw(nL, Hkv, max(Ts), d), draw(nL, m, Hkv * G, d)
        c = cb.CacheBack(nL, Hkv * G, Hkv, d, m, max(Ts), len(Ts), p=p, pool_width=width)
        out, S = [torch.empty(T, device="cuda") for T in Ts], torch.empty(max(Ts), device="cuda")
        c.score([K[:, :, :T] for T in Ts], [Q] * len(Ts), out)
        c.sync_status()
        assert c.score_path() == 2
        for b, T, got in zip(_attention_64(K, Q, Ts), Ts, out):
            assert_scores_close(got.cpu().numpy(), _score_64(b, Hkv, width, p).cpu().numpy(), rtol=RTOL)
            c.score([K[:, :, :T]], [Q], [S[:T]])
            c.sync_status()
            assert torch.equal(S[:T].view(torch.int32), got.view(torch.int32)), (rows, T)


@pytest.mark.parametrize("own", [False, True])
def test_long_chunks(own):
    """1024 groups, enough for chunks of 2048 positions: one with and without a second half, and two;
    the query tokens' own keys join the last."""
    nL, H, d, m, Ts = 64, 16, 64, 5, [130, 1024, 1030, 2049]
    gen = torch.Generator().manual_seed(7)
    draw = lambda *s: torch.randn(*s, generator=gen).bfloat16()
    K, Q, own_k = draw(nL, H, max(Ts), d), draw(nL, m, H, d), draw(nL, m, H, d) if own else None
    c = cb.CacheBack(nL, H, H, d, m, max(Ts), len(Ts))
    Kd, Qd = K.cuda(), Q.cuda()
    out = [torch.empty(T, device="cuda") for T in Ts]
    c.score([Kd[:, :, :T] for T in Ts], [Qd] * len(Ts), out, Kselfs=None if not own else [own_k.cuda()] * len(Ts))
    c.sync_status()
    assert c.score_path() == 2
    for T, got in zip(Ts, out):
        ref = oracle_scores(oracle.default(), K[:, :, :T].contiguous(), Q, Kself=own_k)
        assert_scores_close(got.cpu().numpy(), ref["S"], rtol=RTOL)


def test_senders_of_different_query_lengths_equal_single_calls():
    """Row-chunk counts that differ within a call: every pair's scores are those of its own call."""
    ms, T = [40, 300, 129, 64], [500, 333, 1100, 7]
    w = [synth.custom_workload(synth.Shape(1, 8, 2, 128), [t], m, seed=m, n_planted_spans=1) for t, m in zip(T, ms)]
    Ks, Qs = [x.senders[0].K.cuda() for x in w], [x.queries[0].cuda() for x in w]
    c = make_cb(w[0].spec.shape, max(T), max(ms), len(T))
    out = [torch.empty(t, device="cuda") for t in T]
    c.score(Ks, Qs, out)
    c.sync_status()
    assert c.score_path() == 2
    for i in range(len(T)):
        one = make_cb(w[0].spec.shape, T[i], ms[i], 1)
        S = torch.empty(T[i], device="cuda")
        one.score([Ks[i]], [Qs[i]], [S])
        one.sync_status()
        assert torch.equal(S.view(torch.int32), out[i].view(torch.int32)), i


def test_small_senders_beside_large_ones():
    """Head dimension 64: a call's small senders take the mma.sync passes and the others the tcgen05
    passes; each gets the scores of a call of its own, whichever others are in the call."""
    Ts, m = [200, 4000, 65, 3000], 60
    w = [synth.custom_workload(synth.Shape(4, 16, 8, 64), [t], m, seed=t, n_planted_spans=1) for t in Ts]
    Ks, Qs = [x.senders[0].K.cuda() for x in w], [x.queries[0].cuda() for x in w]
    c = make_cb(w[0].spec.shape, max(Ts), m, len(Ts))
    out = [torch.empty(t, device="cuda") for t in Ts]
    c.score(Ks, Qs, out)
    c.sync_status()
    paths = []
    for i in range(len(Ts)):
        one = make_cb(w[0].spec.shape, Ts[i], m, 1)
        S = torch.empty(Ts[i], device="cuda")
        one.score([Ks[i]], [Qs[i]], [S])
        one.sync_status()
        paths.append(one.score_path())
        assert torch.equal(S.view(torch.int32), out[i].view(torch.int32)), i
        ref = oracle_scores(oracle.default(), w[i].senders[0].K, w[i].queries[0])["S"]
        assert_scores_close(S.cpu().numpy(), ref, rtol=RTOL)
    assert paths == [1, 2, 1, 2] and c.score_path() == 2


def test_position_major_strides():
    """K as [T][nL][Hkv][d] with rows past the last position belonging to nothing."""
    w = synth.custom_workload(synth.Shape(2, 8, 2, 64), [483], 70, seed=3, n_planted_spans=2)
    K, Q = w.senders[0].K.cuda(), w.queries[0].cuda()
    Kp = K.permute(2, 0, 1, 3).contiguous().permute(1, 2, 0, 3)
    out = [torch.empty(483, device="cuda") for _ in range(2)]
    for k, o in zip((K, Kp), out):
        c = make_cb(w.spec.shape, 483, 70, 1)
        c.score([k], [Q], [o])
        c.sync_status()
        assert c.score_path() == 2
    assert torch.equal(out[0].view(torch.int32), out[1].view(torch.int32))


def _paged(K, P, seed):
    nL, Hkv, T, d = K.shape
    n = -(-T // P)
    g = torch.Generator().manual_seed(seed)
    table = torch.randperm(n + 3, generator=g)[:n].to(torch.int32).cuda()
    pool = torch.full((nL, n + 3, P, Hkv, d), float("nan"), dtype=K.dtype, device="cuda")
    full = torch.full((nL, n * P, Hkv, d), float("nan"), dtype=K.dtype, device="cuda")   # rows past T
    full[:, :T] = K.permute(0, 2, 1, 3)
    pool[:, table.long()] = full.view(nL, n, P, Hkv, d)
    return cb.PagedKV(pool, pool, table, T)


@pytest.mark.parametrize("d,m,P", [(64, 70, 16), (128, 200, 16), (128, 40, 8), (128, 40, 128), (64, 300, 512), (128, 20, 4)])
def test_paged_equals_strided(d, m, P):
    """Pages of 8 rows and more go through pass 1's own loads and stores (one box a page, or 128 rows
    of a longer one), shorter ones through the copy kernel."""
    w = synth.custom_workload(synth.Shape(2, 8, 2, d), [1100, 300], m, seed=d, n_planted_spans=2)
    Ks, Q = [s.K.cuda() for s in w.senders], w.queries[0].cuda()
    out = [[torch.empty(t, device="cuda") for t in (1100, 300)] for _ in range(2)]
    for caches, o in zip((Ks, [_paged(K, P, i) for i, K in enumerate(Ks)]), out):
        c = make_cb(w.spec.shape, 1100, m, 2)
        c.score(caches, [Q, Q], o)
        c.sync_status()
        assert c.score_path() == 2
    for a, b in zip(*out):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))


@pytest.mark.parametrize("d,P", [(64, 16), (128, 16), (128, 4)])
def test_paged_with_own_keys_equals_strided(d, P):
    """The query tokens' own keys after the pages' tiles of a group's last chunk."""
    w = synth.custom_workload(synth.Shape(2, 8, 2, d), [1030, 257], 130, seed=d + 1, n_planted_spans=2)
    Ks, Q = [s.K.cuda() for s in w.senders], w.queries[0].cuda()
    own = synth.make_query_keys(w.spec, 5, 0)
    out = [[torch.empty(t, device="cuda") for t in (1030, 257)] for _ in range(2)]
    for caches, o in zip((Ks, [_paged(K, P, i) for i, K in enumerate(Ks)]), out):
        c = make_cb(w.spec.shape, 1030, 130, 2)
        c.score(caches, [Q, Q], o, Kselfs=[own.cuda()] * 2)
        c.sync_status()
        assert c.score_path() == 2
    for i, (a, b) in enumerate(zip(*out)):
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
        ref = oracle_scores(oracle.default(), w.senders[i].K, w.queries[0], Kself=own)["S"]
        assert_scores_close(a.cpu().numpy(), ref, rtol=RTOL)


def test_paged_first_call_inside_a_capture():
    """Shapes that used to read pages directly allocate nothing inside a stream capture: the first
    call there runs the mma.sync passes, and a later one outside the tcgen05 passes."""
    w = synth.custom_workload(synth.Shape(1, 8, 2, 64), [500], 70, seed=4, n_planted_spans=2)
    K, Q = w.senders[0].K.cuda(), w.queries[0].cuda()
    pk = _paged(K, 16, 1)
    c = make_cb(w.spec.shape, 500, 70, 1)
    S = torch.zeros(500, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        c.score([pk], [Q], [S])
    assert c.score_path() == 1
    g.replay()
    torch.cuda.synchronize()
    ref = oracle_scores(oracle.default(), w.senders[0].K, w.queries[0])["S"]
    assert_scores_close(S.cpu().numpy(), ref, rtol=RTOL)
    c.score([pk], [Q], [S])
    c.sync_status()
    assert c.score_path() == 2
    assert_scores_close(S.cpu().numpy(), ref, rtol=RTOL)
