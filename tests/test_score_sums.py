"""The scoring pass's fp32 sums, bit for bit: how many terms a sum has decides how far the scores are from their exact
values, so the order is followed here with numpy.  All tokens sit at position (0, 0, 0), where the rotation is the identity."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2601_04359_b200 import binding as pc

pytestmark = pytest.mark.gpu
F = np.float32


def _inputs(shape, dtype, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(shape, generator=g).to(dtype)


def _scores(q, k, n_kv):
    n_q, n_heads, d = q.shape
    n = len(k)
    ctx = pc.Context(n_heads, n_kv, d, pc.PC_BF16 if q.dtype == torch.bfloat16 else pc.PC_F32, 10000.0, (4, 4, 4), n_q, n)
    zero = lambda m: torch.zeros(m, 4, dtype=torch.int32, device="cuda")
    cache = pc.Cache(pc.Segment.empty(), pc.Segment(k.cuda(), k.cuda(), zero(n), n), np.array([n], np.int32))
    out, _ = pc.pc_score(ctx, cache, q.cuda(), zero(n_q), np.array([1], np.int32))
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    ctx.close()
    return out.cpu().numpy()


def _pooled(sums, n_q):
    """What the scoring kernel makes of the accumulator's fixed-point sums."""
    fx = np.rint(sums.astype(np.float64) * 2.0 ** 32).astype(np.int64).sum(0)
    return (fx.astype(np.float64) * (1.0 / (2.0 ** 32 * n_q))).astype(F)


# (query heads, KV heads, d), tokens in one fp32 sum: 8 warps' worth of a query row cut into warps of up to 4 x 32 chunks
@pytest.mark.parametrize("heads,dtype,tokens", [((24, 8, 128), torch.bfloat16, 2), ((32, 8, 128), torch.bfloat16, 2), ((8, 8, 128), torch.bfloat16, 8),
                                                ((64, 8, 128), torch.bfloat16, 1), ((4, 2, 64), torch.float32, 8), ((8, 4, 128), torch.float32, 4)])
@pytest.mark.parametrize("n_q", [1, 7, 290])               # no more than one token per thread on 148 SMs
def test_pooled_query_is_summed_over_few_tokens(heads, dtype, tokens, n_q):
    hq, hk, d = heads
    q = _inputs((n_q, hq, d), dtype, 1)
    k = torch.eye(hk * d).view(hk * d, hk, d).to(dtype)                # key e reads element e of the pooled query
    x = q.float().numpy().reshape(n_q, hk, hq // hk, d)
    x = np.concatenate([x, np.zeros(((-n_q) % tokens,) + x.shape[1:], F)]).reshape(-1, tokens, hk, hq // hk, d)
    sums = np.zeros((len(x), hk, d), F)
    for w in range(tokens):
        for h in range(hq // hk):
            sums += x[:, w, :, h]
    scale = F(1.0 / (hq * np.sqrt(float(d))))
    assert np.array_equal(_scores(q, k, hk), (_pooled(sums, n_q) * scale).ravel())


@pytest.mark.parametrize("heads,dtype", [((8, 8, 128), torch.bfloat16), ((24, 8, 128), torch.bfloat16), ((4, 2, 64), torch.float32)])
def test_pooled_query_keeps_small_terms_beside_a_large_one(heads, dtype):
    """60,000 tokens of ones and one of 2^24, in which a one added on its own is lost.  A thread walks dozens of tokens; what an
    element may lose is half a spacing (1) for each of the up to 16 terms of the one fp32 sum that the large token is in, half
    a spacing of the result (2^24 / n_q as fp32, 1 in these units, twice) and of the scores' own scale."""
    hq, hk, d = heads
    n_q = 60_000
    q = torch.ones((n_q, hq, d), dtype=dtype)
    q[0] = 2.0 ** 24
    k = torch.eye(hk * d).view(hk * d, hk, d).to(dtype)
    exact = (hq // hk) * (2.0 ** 24 + n_q - 1)
    got = _scores(q, k, hk).astype(np.float64) * hq * np.sqrt(float(d)) * n_q
    assert np.abs(got - exact).max() <= 16 + 3 * (hq // hk)


@pytest.mark.parametrize("n_kv,d,dtype", [(4, 128, torch.bfloat16), (8, 128, torch.bfloat16), (16, 128, torch.bfloat16), (2, 64, torch.float32),
                                          (8, 64, torch.float32), (4, 128, torch.float32), (8, 128, torch.float32)])
@pytest.mark.parametrize("n", [61, 4099])
def test_a_key_is_summed_in_short_chains(n_kv, d, dtype, n):
    q, k = _inputs((1, n_kv, d), dtype, 2), _inputs((n, n_kv, d), dtype, 3)
    per = 8 if dtype == torch.bfloat16 else 4                          # elements of a 16-byte chunk
    lanes = max(16, d // per)                                          # lanes that share a key
    chains = 32 // lanes
    p = _pooled(q.float().numpy().reshape(1, -1), 1).reshape(-1, chains, lanes, per)
    x = k.float().numpy().reshape(n, -1, chains, lanes, per)
    a = np.zeros(x.shape[:1] + x.shape[2:], F)
    for g in range(x.shape[1]):                                        # one rounding per multiply-add: 48 + 24 bits fit a long double closely enough
        a = (p[g].astype(np.longdouble) * x[:, g].astype(np.longdouble) + a.astype(np.longdouble)).astype(F)
    r = np.zeros((n, chains, lanes), F)
    for u in range(per // 2):
        r = (a[..., 2 * u] + a[..., 2 * u + 1]) + r
    s = r[:, 0] + r[:, 1] if chains == 2 else r[:, 0]
    o = lanes // 2
    while o:
        s = s + s[:, np.arange(lanes) ^ o]
        o //= 2
    assert np.array_equal(_scores(q, k, n_kv), s[:, 0] * F(1.0 / (n_kv * np.sqrt(float(d)))))
