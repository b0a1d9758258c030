"""The window step from host memory by its two routes, a kernel that reads pinned memory and the runtime's copies (which pageable
memory takes), on both sides of the rule that chooses: the same regimes, caches and outputs, bit for bit."""
from __future__ import annotations

from dataclasses import replace

import pytest
import torch

from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import workload as wl
from paper_2601_04359_b200.device import DeviceLayer, make_ctx

pytestmark = pytest.mark.gpu


# 24 / 8 heads: 383 tokens move 6.27 MB, the last size below 6 MiB of one part; 4 / 2 fp32 heads of 64
@pytest.mark.parametrize("grid,heads,dtype,d", [((1, 1), (24, 8), wl.BF16, 128), ((9, 15), (24, 8), wl.BF16, 128), ((1, 383), (24, 8), wl.BF16, 128),
                                                ((12, 32), (24, 8), wl.BF16, 128), ((8, 8), (4, 2), wl.F32, 64)])
def test_pinned_and_pageable_memory_give_the_same_step(grid, heads, dtype, d):
    cfg = replace(wl.small_bf16(n_frames=3, grid=grid, n_text=5, total=max(2, int(1.4 * grid[0] * grid[1])), kind=wl.LINEAR, param=0.0, keep_full=0, seed=3),
                  n_q_heads=heads[0], n_kv_heads=heads[1], dtype=dtype, head_dim=d)
    n, total = cfg.frame_tokens, cfg.budget.total
    D = DeviceLayer(wl.make_layer(cfg, with_current=True))
    h, cap = D.cache.history, total + 2 * n
    mk = lambda: pc.Segment(torch.zeros((cap,) + h.k.shape[1:], dtype=h.k.dtype, device="cuda"), torch.zeros((cap,) + h.k.shape[1:], dtype=h.k.dtype, device="cuda"),
                            torch.zeros((cap, 4), dtype=torch.int32, device="cuda"), 0)
    ctxs = [make_ctx(cfg, max_keys=cfg.n_anchor + cap) for _ in range(2)]
    wins = [pc.Window(c, 2, pc.PC_LINEAR, 0.0, total, 0, D.cache.anchors, mk(), mk()) for c in ctxs]
    ws = [{"q": torch.zeros_like(D.q), "q_pos": torch.zeros_like(D.q_pos), "out": torch.zeros_like(D.q)} for _ in range(2)]
    homes = [torch.empty(D.q.shape, dtype=D.q.dtype).pin_memory(), torch.empty(D.q.shape, dtype=D.q.dtype)]
    for f in range(4):
        k, v, pos = (x[(f % 3) * n:(f % 3 + 1) * n].cpu().contiguous() for x in (h.k, h.v, h.pos))
        regimes = []
        for i, put in enumerate((lambda x: x.pin_memory(), lambda x: x)):
            homes[i].fill_(9.0)
            frame = {"k": put(k), "v": put(v), "pos": put(pos)} if f < 3 else None         # the last step appends nothing
            regimes.append(wins[i].step_host(frame, put(D.q.cpu()), put(D.q_pos.cpu()), homes[i], ws[i]))
            assert pc.pc_poll_status(ctxs[i]) == pc.PC_OK
        assert regimes[0] == regimes[1] and torch.equal(*homes) and torch.equal(homes[0], ws[0]["out"].cpu())
        assert torch.equal(ws[0]["q"].cpu(), D.q.cpu()) and torch.equal(ws[0]["q_pos"].cpu(), D.q_pos.cpu())
        a, b = (w.cache().history for w in wins)
        m = a.n_tokens
        assert m == b.n_tokens and all(torch.equal(x[:m], y[:m]) for x, y in ((a.k, b.k), (a.v, b.v), (a.pos, b.pos)))
    for x in wins + ctxs:
        x.close()
