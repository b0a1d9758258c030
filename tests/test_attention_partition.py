"""The persistent attention kernel's division of (item, key tile) steps over its CTAs, at the counts where the division
changes: one CTA per SM, a few less so that runs line up, one item cut into several parts, a run of whole items."""
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


# 520 query rows of 24 / 8 heads are 64 items of two query tiles.  Of 148 CTAs: 3 key tiles (two steps a run with 148 or
# 144 CTAs: 144), 23 (ten steps with 148, eleven with 144: 148), 37 (sixteen or seventeen: 148); 1 key tile (64 CTAs)
@pytest.mark.parametrize("n_keys", [3 * 128 - 5, 23 * 128, 37 * 128 + 1 - 128, 100])
def test_attention_over_run_lengths(n_keys):
    _attend((24, 8), (20, 26), n_keys)


# a few items of several key tiles: every item cut into 1, 2, 5, 7 or 8 ranges of its own (a merge of more than four parts
# runs in two rounds), one more tile than ranges, and an item's last range of a single key
@pytest.mark.parametrize("heads,grid,n_keys", [((8, 8), (1, 100), 128), ((8, 8), (1, 100), 256), ((8, 8), (1, 100), 5 * 128), ((8, 8), (3, 47), 7 * 128),
                                               ((8, 8), (1, 100), 8 * 128 + 1), ((2, 2), (9, 15), 40 * 128), ((16, 4), (10, 20), 11 * 128 - 1),
                                               ((24, 12), (14, 26), 11 * 128)])
def test_attention_with_few_items(heads, grid, n_keys):
    _attend(heads, grid, n_keys)


def _attend(heads, grid, n_keys):
    hq, hkv = heads
    cfg = replace(wl.small_bf16(n_frames=1, grid=grid, n_text=1, seed=90), outliers=False, n_q_heads=hq, n_kv_heads=hkv)
    L = wl.make_layer(cfg)
    rng = np.random.default_rng(n_keys)
    L.hist_k, L.hist_v = (wl.round_bf16(rng.standard_normal((n_keys, hkv, 128)).astype(np.float32)) for _ in range(2))
    L.hist_pos = np.stack([np.arange(n_keys) % 10, np.arange(n_keys) % cfg.max_pos[1], np.arange(n_keys) % cfg.max_pos[2], np.arange(n_keys)], axis=1).astype(np.int32)
    L.frame_count = np.array([n_keys], np.int32)
    L.anchor_k, L.anchor_v, L.anchor_pos = L.anchor_k[:0], L.anchor_v[:0], L.anchor_pos[:0]
    D = DeviceLayer(L)
    ctx = make_ctx(cfg, max_keys=n_keys)
    out, lse = pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos, want_lse=True)
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    # two rows of every (row tile, head)
    rows = np.array([(min(t * 128 + int(rng.integers(128)), cfg.n_q - 1), h) for t in range((cfg.n_q + 127) // 128) for h in range(hq) for _ in range(2)], np.int32)
    segs = [(L.hist_k, L.hist_v, L.hist_pos)]
    want, want_lse = oracle.attend(L.q, L.q_pos, segs, rows=rows, want_lse=True)
    got = host(out)[rows[:, 0], rows[:, 1]].astype(np.float64)
    assert attention_within_bounds(got, want, oracle.attend(L.q, L.q_pos, abs_v(segs), rows=rows))
    assert np.abs(host(lse)[rows[:, 0], rows[:, 1]] - want_lse).max() <= 2e-2
    ctx.close()
