"""The query pass at the token counts where its division changes: fewer tokens than a block's slots, one block more, one
round of the persistent grid and one token past it, several rounds; and its accumulator, which the scoring kernel clears."""
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


@pytest.mark.parametrize("heads,dtype,d", [((24, 8), wl.BF16, 128), ((32, 8), wl.BF16, 128), ((4, 2), wl.F32, 64)])
@pytest.mark.parametrize("n_q", [1, 3, 5, 592, 593, 1999])
def test_pooled_query_over_token_counts(heads, dtype, d, n_q):
    cfg = replace(wl.small_bf16(n_frames=1, grid=(1, n_q), n_text=4, total=1, keep_full=0, seed=n_q), n_q_heads=heads[0], n_kv_heads=heads[1],
                  dtype=dtype, head_dim=d)
    L = wl.make_layer(cfg)
    D = DeviceLayer(L)
    ctx = make_ctx(cfg)
    zero = np.zeros(1, np.int32)
    ref = oracle.score_pooled(L.hist_k, L.hist_pos, L.q, L.q_pos)
    scores, _ = pc.pc_score(ctx, D.cache, D.q, D.q_pos, zero)
    assert (np.abs(host(scores).astype(np.float64) - ref) <= score_tolerance(ref, L.frame_count)).all()
    again, _ = pc.pc_score(ctx, D.cache, D.q, D.q_pos, zero)           # the accumulator was zero again, and sums repeat bit for bit
    assert torch.equal(scores, again) and pc.pc_poll_status(ctx) == pc.PC_OK
    ctx.close()
