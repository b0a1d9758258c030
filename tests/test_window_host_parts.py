"""The window step from host memory at the frame sizes where attention runs in one part, in two, and in parts of unequal
size, against the device-side step on a second window: the cache bit for bit; the output of one part, too, that of several
within what other cuts of the keys can move it.  A cut moves the reference that a row's probabilities are taken against, and
with it their bf16 rounding, 2^-9 relative each on either side and independent from key to key: 2 * 2^-9 * max|v| *
sqrt(sum p^2), with |v| up to 5 (outlier channels of 4 and noise) and sqrt(sum p^2) below 0.1 from a thousand keys of
unit-variance logits on; 2e-3 and one spacing of bf16 numbers for storing the results."""
from __future__ import annotations

from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import workload as wl
from paper_2601_04359_b200.device import DeviceLayer, make_ctx

from .test_gpu_parity import bf16_ulp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(7, 9), (16, 16), (20, 26), (24, 42), (33, 40), (40, 64)])
def test_host_step_in_parts(grid):
    _check(grid, (24, 8), grid[0] * grid[1] <= 256, 2e-3)


@pytest.mark.parametrize("grid,heads,one_part", [((16, 24), (24, 8), True), ((5, 77), (24, 8), False), ((8, 16), (64, 8), True), ((3, 43), (64, 8), False)])
def test_host_step_at_the_last_row_of_one_part(grid, heads, one_part):
    """384 and 385 rows of 24 / 8 heads, 128 and 129 of 64 / 8: where one part becomes two on 148 SMs.  With a few hundred keys
    a single probability can be large, so the bound is 2 * 2^-9 * sum p |v| <= 2^-8 max|v|."""
    _check(grid, heads, one_part and torch.cuda.get_device_properties(0).multi_processor_count == 148, None)


def _check(grid, heads, one_part, bound):
    cfg = replace(wl.small_bf16(n_frames=3, grid=grid, n_text=37, total=int(1.3 * grid[0] * grid[1]), kind=wl.LINEAR, param=0.0, keep_full=0, seed=7),
                  n_q_heads=heads[0], n_kv_heads=heads[1])
    n, W, total = cfg.frame_tokens, 2, cfg.budget.total
    D = DeviceLayer(wl.make_layer(cfg, with_current=True))
    h = D.cache.history
    cap = total + 2 * n
    shape = (cap, cfg.n_kv_heads, cfg.head_dim)
    mk = lambda: pc.Segment(torch.zeros(shape, dtype=torch.bfloat16, device="cuda"), torch.zeros(shape, dtype=torch.bfloat16, device="cuda"),
                            torch.zeros((cap, 4), dtype=torch.int32, device="cuda"), 0)
    ctxs = [make_ctx(cfg, max_keys=cfg.n_anchor + cap) for _ in range(2)]
    wins = [pc.Window(c, W, pc.PC_LINEAR, 0.0, total, 0, D.cache.anchors, mk(), mk()) for c in ctxs]
    ws = {"q": torch.empty_like(D.q), "q_pos": torch.empty_like(D.q_pos), "out": torch.empty_like(D.q)}
    out_host = torch.empty(D.q.shape, dtype=torch.bfloat16).pin_memory()
    pin = lambda x: x.cpu().pin_memory()
    for f in range(3):
        k, v, pos = (x[f * n:(f + 1) * n].contiguous() for x in (h.k, h.v, h.pos))
        wins[0].append(pc.Segment(k, v, pos, n))
        regime, out = wins[0].step(D.q, D.q_pos)
        out_host.fill_(9.0)
        assert wins[1].step_host({"k": pin(k), "v": pin(v), "pos": pin(pos)}, pin(D.q), pin(D.q_pos), out_host, ws) == regime
        assert all(pc.pc_poll_status(c) == pc.PC_OK for c in ctxs)
        a, b = (w.cache().history for w in wins)
        m = a.n_tokens
        assert m == b.n_tokens and all(torch.equal(x[:m], y[:m]) for x, y in ((a.k, b.k), (a.v, b.v), (a.pos, b.pos)))
        got, want = out_host.float().numpy(), out.float().cpu().numpy()
        assert (np.abs(got - want) <= bf16_ulp(want) + (bound or 2.0 ** -8 * float(torch.cat([D.cache.anchors.v, a.v[:m]]).float().abs().max()))).all()
        if one_part:
            assert torch.equal(out_host, out.cpu())
    for w in wins:
        w.close()
    for c in ctxs:
        c.close()
