"""Keys past a segment's end in its last tile: they are masked in columns of eight and single ones, one tile per segment at
least, in a run's first step (whose scores of the second query tile lie elsewhere) and in later ones."""
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


# keys of the anchors and of the history: one tile each, two and three, remainders 1, 7, 8, 9, 120, 121, 127 and 0
@pytest.mark.parametrize("n_anchor,n_hist", [(1, 127), (7, 121), (8, 120), (9, 128), (128, 1), (129, 137), (255, 264), (256, 300), (376, 9)])
@pytest.mark.parametrize("grid", [(1, 5), (11, 13)])
def test_keys_past_a_segments_end_have_no_weight(n_anchor, n_hist, grid):
    cfg = replace(wl.small_bf16(n_frames=1, grid=grid, n_text=1, seed=91), outliers=False)
    L = wl.make_layer(cfg)
    rng = np.random.default_rng(1000 * n_anchor + n_hist)

    def seg(n):
        k, v = (wl.round_bf16(rng.standard_normal((n, cfg.n_kv_heads, 128)).astype(np.float32)) for _ in range(2))
        i = np.arange(n)
        return k, v, np.stack([i % 10, i % cfg.max_pos[1], i % cfg.max_pos[2], i], axis=1).astype(np.int32)

    L.anchor_k, L.anchor_v, L.anchor_pos = seg(n_anchor)
    L.hist_k, L.hist_v, L.hist_pos = seg(n_hist)
    L.frame_count = np.array([n_hist], np.int32)
    D = DeviceLayer(L)
    ctx = make_ctx(cfg, max_keys=n_anchor + n_hist)
    out, lse = pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos, want_lse=True)
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    rows = np.array([(int(rng.integers(cfg.n_q)), h) for h in range(cfg.n_q_heads) for _ in range(4)], np.int32)
    segs = [(L.anchor_k, L.anchor_v, L.anchor_pos), (L.hist_k, L.hist_v, L.hist_pos)]
    want, want_lse = oracle.attend(L.q, L.q_pos, segs, rows=rows, want_lse=True)
    assert attention_within_bounds(host(out)[rows[:, 0], rows[:, 1]].astype(np.float64), want, oracle.attend(L.q, L.q_pos, abs_v(segs), rows=rows))
    assert np.abs(host(lse)[rows[:, 0], rows[:, 1]] - want_lse).max() <= 2e-2      # the bf16 bound on log-sum-exps
    ctx.close()
