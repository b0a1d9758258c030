"""The CUDA-core attention kernel at the edges of its tiles (32 keys, 32 or 64 rows of a KV head's group) and key ranges,
against the oracle: one key, a tile less one, a tile, a tile more, several ranges; both head dimensions and types."""
from __future__ import annotations

from dataclasses import replace

import numpy as np
import pytest

import oracle
from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import workload as wl
from paper_2601_04359_b200.device import DeviceLayer, host, make_ctx

from .test_randomized_shapes import abs_v, attention_within_bounds

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,heads", [(wl.F32, 64, (4, 2)), (wl.F32, 128, (6, 2)), (wl.BF16, 64, (3, 1)), (wl.BF16, 128, (5, 5))])
@pytest.mark.parametrize("n_keys,grid", [(1, (1, 1)), (31, (3, 7)), (32, (4, 8)), (33, (1, 33)), (257, (5, 13)), (300, (40, 50))])
def test_cuda_core_attention_at_tile_edges(dtype, d, heads, n_keys, grid):
    cfg = replace(wl.small_bf16(n_frames=1, grid=grid, n_text=2, seed=60), n_q_heads=heads[0], n_kv_heads=heads[1], head_dim=d, dtype=dtype,
                  outliers=False)
    L = wl.make_layer(cfg)
    rng = np.random.default_rng(n_keys)
    n_anchor = n_keys // 3                                             # a second segment wherever there are keys for it
    draw = lambda n: wl.to_storage(rng.standard_normal((n, heads[1], d)).astype(np.float32), dtype)
    pos = np.stack([np.arange(n_keys) % 8, np.arange(n_keys) % min(cfg.max_pos[1], 50), np.arange(n_keys) % min(cfg.max_pos[2], 50),
                    np.arange(n_keys)], axis=1).astype(np.int32)
    L.anchor_k, L.anchor_v, L.anchor_pos = draw(n_anchor), draw(n_anchor), pos[:n_anchor]
    L.hist_k, L.hist_v, L.hist_pos = draw(n_keys - n_anchor), draw(n_keys - n_anchor), pos[n_anchor:]
    L.frame_count = np.array([n_keys - n_anchor], np.int32)
    D = DeviceLayer(L)
    ctx = make_ctx(cfg, max_keys=n_keys)
    pc.pc_set_attend_impl(ctx, 1)
    out, lse = pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos, want_lse=True)
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    rows = np.array([(i, h) for i in range(0, cfg.n_q, max(1, cfg.n_q // 70)) for h in range(heads[0])] +
                    [(cfg.n_q - 1, heads[0] - 1)], np.int32)
    segs = [s for s in [(L.anchor_k, L.anchor_v, L.anchor_pos), (L.hist_k, L.hist_v, L.hist_pos)] if len(s[0])]
    want, want_lse = oracle.attend(L.q, L.q_pos, segs, cfg.rope_base, rows=rows, want_lse=True)
    got = host(out)[rows[:, 0], rows[:, 1]].astype(np.float64)
    if dtype == wl.F32:
        assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()
        assert np.abs(host(lse)[rows[:, 0], rows[:, 1]] - want_lse).max() <= 1e-4
    else:
        assert attention_within_bounds(got, want, oracle.attend(L.q, L.q_pos, abs_v(segs), cfg.rope_base, rows=rows))
    assert np.isfinite(host(out)).all()
    ctx.close()
