"""Errors of scores against 64 bits: the tcgen05 passes are no less exact than the mma.sync passes.

Both contract bf16 inputs with 32-bit sums; they differ in where a row's offset is subtracted and in
how the tensor core rounds its sums.  The error is the 2-norm of the difference over that of the
scores, averaged over several inputs; it is a few 1e-7 on either path.
"""
import math

import pytest
import torch

import synth
from gpu_helpers import make_cb

pytestmark = pytest.mark.gpu


def _scores_64(K, Q, alpha, pool=7):
    """Scores at p = 2 in 64 bits, by their definition."""
    nL, Hkv, T, d = K.shape
    m, Hq = Q.shape[1:3]
    G = Hq // Hkv
    widest = lambda x: torch.nn.functional.max_pool1d(x.view(1, -1, T), pool, 1, pool // 2).view(x.shape)
    U = N = D = 0
    for l in range(nL):
        for g in range(Hkv):
            q = Q[l, :, g * G:(g + 1) * G].double().reshape(m * G, d)
            b = torch.softmax(q @ K[l, g].double().T / math.sqrt(d), -1).view(m, G, T).mean(1)
            U = U + b.mean(0) / Hkv
            N = N + (widest(b) ** 2).mean(0)
            D = D + widest(b.mean(0)) ** 2
    return widest(U) * (N / D) ** alpha


@pytest.mark.parametrize("alpha", [0.0, 2.0])
@pytest.mark.parametrize("d,m", [(64, 70), (128, 40), (128, 140)])
def test_tcgen05_no_less_exact_than_mma_sync(d, m, alpha):
    shape, T, seeds = synth.Shape(8, 16, 4, d), 3001, 6
    errs = {1: 0.0, 2: 0.0}
    for seed in range(seeds):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        draw = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
        K, Q, S = draw(8, 4, T, d), draw(8, m, 16, d), torch.empty(T, device="cuda")
        ref = _scores_64(K, Q, alpha)
        for kernel in errs:
            c = make_cb(shape, T, m, 1, alpha=alpha, score_kernel=kernel % 2)
            c.score([K], [Q], [S])
            c.sync_status()
            assert c.score_path() == kernel
            errs[kernel] += float((S.double() - ref).norm() / ref.norm()) / seeds
    assert errs[2] <= errs[1], errs
