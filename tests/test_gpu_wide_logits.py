"""Rows of attention whose logits spread widely, on the tcgen05 score passes.

Pass 1 keeps, per row and quarter of a chunk of positions, an offset and the sum of exp2 of the
logits above it; the combine kernel brings all of a row's partials to one offset.  A row's largest
logits may lie far above the first logits of their partial, and in other partials than the largest
offset: the result must be right, and take no longer than for other logits.

Tolerance: a logit of up to 150 (log2 domain) is a 32-bit sum of d / 16 tensor-core steps, each off
by up to an ulp of it, 2^-16 of 150 in units of log2: 1e-5 of the exponential a step, 1e-4 for all.
A score is a mean of exponentials times the square of a ratio of such means: 3e-4, well within the
2e-3 of the score parity tests; the fault this guards against is off by 0.1 and more.
"""
import math

import pytest
import torch

import oracle
import paper_2609_32046_gb300 as cb
import synth
from gpu_helpers import assert_scores_close, make_cb, oracle_scores

pytestmark = pytest.mark.gpu

RTOL = 5e-4
T, M, ROW, HEAD = 2049, 70, 35, 5        # the last chunk of 1024 positions has one position
NEEDLE = 3 * 128 + 5                      # chunk 0, column quarter 0 (positions 0-31 of every 128)
OTHER = {"quarter": 32, "chunk": 1024}    # first position of another quarter's, another chunk's partial


def _pages(K, P=16):
    """K in pages of P positions in a random order; rows past T hold NaN."""
    nL, Hkv, n_pos, d = K.shape
    n = -(-n_pos // P)
    table = torch.randperm(n + 3, generator=torch.Generator().manual_seed(1))[:n].to(torch.int32).cuda()
    pool = torch.full((nL, n + 3, P, Hkv, d), float("nan"), dtype=K.dtype, device="cuda")
    full = torch.full((nL, n * P, Hkv, d), float("nan"), dtype=K.dtype, device="cuda")
    full[:, :n_pos] = K.permute(0, 2, 1, 3)
    pool[:, table.long()] = full.view(nL, n, P, Hkv, d)
    return cb.PagedKV(pool, pool, table, n_pos)


# gap: the needle's logit above that of the low positions that open its partial; exp2 of it leaves
# 32-bit range from 128 on, and exp2 of its negative from 126 on.
@pytest.mark.parametrize("paged", [False, True], ids=["strided", "paged"])
@pytest.mark.parametrize("other", ["quarter", "chunk", "own"])
@pytest.mark.parametrize("low", [1, 32], ids=["low_first", "low_block"])
@pytest.mark.parametrize("d", [64, 128])
def test_needles_far_above_their_partials_offset(d, low, other, paged):
    shape = synth.Shape(1, 8, 2, d)
    w = synth.custom_workload(shape, [T], M, seed=d, n_planted_spans=0)
    K0, Q = w.senders[0].K, w.queries[0]
    own0 = synth.make_query_keys(w.spec, 5, 0) if other == "own" else None
    g, q = HEAD // 4, Q[0, ROW, HEAD].float()
    unit = math.sqrt(d) / (math.log2(math.e) * float(q.norm()))   # |k| of a logit of one (log2 domain)
    key = lambda x: (q / q.norm() * (x * unit)).to(torch.bfloat16)
    base = 0.0 if low == 1 else -30.0
    o = oracle.default()
    c = make_cb(shape, T, M, 1)
    S = torch.empty(T, device="cuda")
    for gap in (100.0, 120.0, 125.5, 126.3, 127.2, 128.5, 130.5, 131.5, 134.0, 142.0):
        K, own = K0.clone(), None if own0 is None else own0.clone()
        K[0, g, :low] = key(base)
        K[0, g, NEEDLE] = key(base + gap)
        if other == "own":
            own[0, 32, g] = key(base + gap - 0.1)   # column quarter 1, which has no position in the last chunk
        else:
            K[0, g, OTHER[other]] = key(base + gap - 0.1)
        Kd = K.cuda()
        c.score([_pages(Kd) if paged else Kd], [Q.cuda()], [S], Kselfs=None if own is None else [own.cuda()])
        c.sync_status()
        assert c.score_path() == 2
        assert_scores_close(S.cpu().numpy(), oracle_scores(o, K, Q, Kself=own)["S"], rtol=RTOL)


@pytest.mark.parametrize("d", [64, 128])
def test_wide_logits_take_no_longer(d):
    """Logits of standard deviation 30 (natural units): the statistics of a row still come from its
    partials (recomputing such rows from Q and K takes milliseconds)."""
    nL, Hq, Hkv, T, m = 8, 16, 4, 2048, 80
    gen = torch.Generator(device="cuda").manual_seed(d)
    draw = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    K, Q, S = draw(nL, Hkv, T, d), draw(nL, m, Hq, d), torch.empty(T, device="cuda")
    c = make_cb(synth.Shape(nL, Hq, Hkv, d), T, m, 1)
    ms = []
    for sd in (1, 30):
        Kd = K * sd
        c.score([Kd], [Q], [S])
        c.enable_stage_timing(True)
        c.stage_times()
        for _ in range(3):
            c.score([Kd], [Q], [S])
        ms.append(c.stage_times()[0])
        c.sync_status()
        c.enable_stage_timing(False)
        assert c.score_path() == 2
        assert_scores_close(S.cpu().numpy(), oracle_scores(oracle.default(), Kd, Q)["S"])
    assert sum(ms[1].values()) < 2 * sum(ms[0].values()) + 0.2, ms
