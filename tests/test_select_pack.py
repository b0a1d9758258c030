"""Selection and pack in one launch: the fused step against the separate calls, bit for bit, on both sides of the rule that
chooses it (frames of 256 and 257 tokens, as many blocks as SMs and more) and around a block's eight ranks."""
from __future__ import annotations

from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import workload as wl
from paper_2601_04359_b200.device import DeviceLayer, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,dtype,d", [((24, 8), wl.BF16, 128), ((4, 2), wl.F32, 64), ((4, 3), wl.F32, 128)])
@pytest.mark.parametrize("n_frames,grid,quota", [(3, (1, 9), (9, 0, 1)), (3, (1, 40), (7, 8, 9)), (2, (16, 16), (256, 255)), (1, (1, 257), (200,)),
                                                 (4, (16, 16), (17, 256, 1, 100)), (5, (16, 16), (240, 30, 1, 16, 8)), (148, (1, 9), (8,) * 148),
                                                 (148, (1, 10), (9,) * 148)])
def test_one_launch_gives_the_bits_of_two(heads, dtype, d, n_frames, grid, quota):
    if heads[0] % heads[1]:
        heads = (heads[1], heads[1])
    cfg = replace(wl.small_bf16(n_frames=n_frames, grid=grid, n_text=5, total=1, keep_full=0, seed=n_frames), n_q_heads=heads[0], n_kv_heads=heads[1],
                  dtype=dtype, head_dim=d)
    L = wl.make_layer(cfg)
    D, ctx, budget = DeviceLayer(L), make_ctx(cfg), np.array(quota, np.int32)
    n_sel = int(budget.sum())
    scores, sel = pc.pc_score(ctx, D.cache, D.q, D.q_pos, budget)
    two = D.empty_packed(n_sel + 3, poison=5.0)
    pc.pc_compact(ctx, D.cache, sel, budget, 4, two)
    out, _ = pc.pc_attend_frame(ctx, two, None, D.q, D.q_pos, want_lse=True)
    one = D.empty_packed(n_sel + 3, poison=5.0)
    sel1 = torch.full((n_sel + 8,), -7, dtype=torch.int32, device="cuda")
    out1 = torch.zeros_like(out)
    pc.pc_frame_step(ctx, D.cache, budget, 4, one, D.q, D.q_pos, scores=torch.zeros_like(scores), sel_idx=sel1[:n_sel], out=out1)
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    assert torch.equal(sel1[:n_sel], sel[:n_sel]) and (sel1[n_sel:] == -7).all()
    for name in ("k", "v", "pos"):
        assert torch.equal(getattr(one.history, name), getattr(two.history, name)), name
    assert torch.equal(out, out1)
    ctx.close()
