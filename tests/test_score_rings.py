"""The scoring kernel at the history lengths where its division changes: less than a warp's group of tokens, a group and a
token, one group for every warp of the grid and a token past it, several turns of the rings; every row width and lane split
(heads of 64 and 128, one or two tokens in a lane)."""
from __future__ import annotations

from dataclasses import replace

import numpy as np
import pytest
import torch

import oracle
from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import workload as wl
from paper_2601_04359_b200.device import DeviceLayer, host, make_ctx, score_tolerance

pytestmark = pytest.mark.gpu

TURN = 148 * 12                                              # warps of the largest grid


# 1 to 4 KB rows; 12 and 16 heads of 128 change from one to two tokens in a lane past TURN pairs of tokens
@pytest.mark.parametrize("heads,dtype,d", [((24, 8), wl.BF16, 128), ((24, 12), wl.BF16, 128), ((16, 16), wl.BF16, 128), ((4, 2), wl.BF16, 128),
                                           ((8, 8), wl.BF16, 64), ((4, 2), wl.F32, 64), ((4, 1), wl.F32, 128), ((8, 8), wl.F32, 128)])
@pytest.mark.parametrize("n", [1, 2, 5, 595, 2 * TURN, 2 * TURN + 1, 4 * TURN + 1, 23001])
def test_scores_over_history_lengths(heads, dtype, d, n):
    cfg = replace(wl.small_bf16(n_frames=1, grid=(1, n), n_text=4, total=1, keep_full=0, seed=n), n_q_heads=heads[0], n_kv_heads=heads[1],
                  dtype=dtype, head_dim=d)
    L = wl.make_layer(cfg)
    D = DeviceLayer(L)
    ctx = make_ctx(cfg)
    q, q_pos = D.q[:40].contiguous(), D.q_pos[:40].contiguous()
    ref = oracle.score_pooled(L.hist_k, L.hist_pos, L.q[:40], L.q_pos[:40])
    zero = np.zeros(1, np.int32)
    out = torch.full((n + 64,), 7.0, device="cuda")
    pc.pc_score(ctx, D.cache, q, q_pos, zero, scores=out[:n])
    assert (np.abs(host(out[:n]).astype(np.float64) - ref) <= score_tolerance(ref, L.frame_count)).all()
    assert (out[n:] == 7.0).all()                            # nothing past the history
    first = out[:n].clone()
    pc.pc_score(ctx, D.cache, q, q_pos, zero, scores=out[:n])
    assert torch.equal(out[:n], first) and pc.pc_poll_status(ctx) == pc.PC_OK
    ctx.close()
