"""The attention mass where its division over CTAs changes: one key tile, an odd number of tiles, units cut into two to four
pieces, runs that cross several units, runs of whole units; each against the oracle, key by key."""
from __future__ import annotations

from dataclasses import replace

import numpy as np
import pytest

import oracle
from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import workload as wl
from paper_2601_04359_b200.device import DeviceLayer, host, make_ctx

from .test_attention_mass import _check_mass

pytestmark = pytest.mark.gpu


# (heads, grid, keys): 2 / 2 heads x 8 query tiles and one pair of key tiles are two units of eight steps on four or five CTAs;
# 24 / 8 heads x 135 queries are units of six steps: 8, 16, 40 and 152 of them; five query heads per KV head units of five
@pytest.mark.parametrize("heads,grid,n_keys", [((2, 2), (25, 40), 100), ((2, 2), (25, 40), 129), ((24, 8), (9, 15), 100), ((24, 8), (9, 15), 385),
                                               ((24, 8), (9, 15), 1200), ((24, 8), (9, 15), 4800), ((6, 2), (1, 1), 257), ((8, 8), (16, 24), 640), ((10, 2), (10, 10), 200)])
def test_mass_over_divisions(heads, grid, n_keys):
    cfg = replace(wl.small_bf16(n_frames=1, grid=grid, n_text=1, seed=91), n_q_heads=heads[0], n_kv_heads=heads[1], outliers=False)
    L = wl.make_layer(cfg)
    rng = np.random.default_rng(n_keys)
    L.hist_k, L.hist_v = (wl.round_bf16(rng.standard_normal((n_keys, heads[1], 128)).astype(np.float32)) for _ in range(2))
    i = np.arange(n_keys)
    L.hist_pos = np.stack([i % 9, i % cfg.max_pos[1], i % cfg.max_pos[2], i], axis=1).astype(np.int32)
    L.frame_count = np.array([n_keys], np.int32)
    L.anchor_k, L.anchor_v, L.anchor_pos = L.anchor_k[:0], L.anchor_v[:0], L.anchor_pos[:0]
    D = DeviceLayer(L)
    ctx = make_ctx(cfg, max_keys=n_keys)
    _, lse = pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos, want_lse=True)
    got = host(pc.pc_attend_mass(ctx, lse, n_keys)).astype(np.float64)
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    _check_mass(got, oracle.attend_mass(L.q, L.q_pos, [(L.hist_k, L.hist_pos)], cfg.rope_base))
    again = host(pc.pc_attend_mass(ctx, lse, n_keys)).astype(np.float64)
    assert np.array_equal(got, again)
    ctx.close()
