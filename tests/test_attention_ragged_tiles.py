"""Keys past a segment's end in its last tile: they are masked in columns of eight and single ones.  One to three key tiles a segment, a
CTA with one step or with a whole item; then runs of a dozen steps that cross from item to item over three segments, of which every
one spans several tiles, and key ranges that begin in any segment."""
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


def _with_segments(cfg, n_anchor, n_hist, seed):
    """A layer with anchors and history of these many keys beside the current frame's."""
    L = wl.make_layer(cfg, with_current=True)
    rng = np.random.default_rng(seed)

    def seg(n):
        k, v = (wl.round_bf16(rng.standard_normal((n, cfg.n_kv_heads, 128)).astype(np.float32)) for _ in range(2))
        i = np.arange(n)
        return k, v, np.stack([i % 10, i % cfg.max_pos[1], i % cfg.max_pos[2], i], axis=1).astype(np.int32)

    L.anchor_k, L.anchor_v, L.anchor_pos = seg(n_anchor)
    L.hist_k, L.hist_v, L.hist_pos = seg(n_hist)
    L.frame_count = np.array([n_hist], np.int32)
    return L, rng


def _check(L, ctx, rng):
    cfg = L.cfg
    D = DeviceLayer(L)
    out, lse = pc.pc_attend_frame(ctx, D.cache, D.current, D.q, D.q_pos, want_lse=True)
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    rows = np.array([(min(t * 128 + int(rng.integers(128)), cfg.n_q - 1), h) for t in range((cfg.n_q + 127) // 128) for h in range(cfg.n_q_heads)
                     for _ in range(2)], np.int32)
    segs = [(L.anchor_k, L.anchor_v, L.anchor_pos), (L.hist_k, L.hist_v, L.hist_pos), (L.cur_k, L.cur_v, L.q_pos)]
    want, want_lse = oracle.attend(L.q, L.q_pos, segs, rows=rows, want_lse=True)
    assert attention_within_bounds(host(out)[rows[:, 0], rows[:, 1]].astype(np.float64), want, oracle.attend(L.q, L.q_pos, abs_v(segs), rows=rows))
    assert np.abs(host(lse)[rows[:, 0], rows[:, 1]] - want_lse).max() <= 2e-2      # the bf16 bound on log-sum-exps
    ctx.close()


# 816 query rows of 24 / 8 heads are 88 items; 19 key tiles: 148 CTAs with 11 or 12 steps each, 22: 148 with boundaries reckoned in.
# Remainders 1, 1 and 48; 44, 3 and 48
@pytest.mark.parametrize("n_anchor,n_hist", [(129, 1153), (300, 1411)])
def test_runs_that_cross_items_and_segments(n_anchor, n_hist):
    cfg = replace(wl.small_bf16(n_frames=1, grid=(24, 34), n_text=1, seed=93), outliers=False)
    L, rng = _with_segments(cfg, n_anchor, n_hist, n_hist)
    _check(L, make_ctx(cfg, max_keys=n_anchor + n_hist + cfg.n_q), rng)


# 143 current keys; ranges of three to eight tiles begin in the first, second or third segment, inside it and on its first tile
@pytest.mark.parametrize("n_anchor,n_hist", [(1, 127), (129, 137), (376, 9), (127, 500)])
@pytest.mark.parametrize("splits,cluster", [(1, False), (2, False), (3, False), (3, True), (4, True)])
def test_key_ranges_that_begin_in_any_segment(n_anchor, n_hist, splits, cluster):
    cfg = replace(wl.small_bf16(n_frames=1, grid=(11, 13), n_text=1, seed=94), outliers=False)
    L, rng = _with_segments(cfg, n_anchor, n_hist, 7 * n_anchor + n_hist)
    ctx = make_ctx(cfg, max_keys=n_anchor + n_hist + cfg.n_q)
    pc.pc_set_kv_splits(ctx, splits)
    pc.pc_set_cluster_merge(ctx, cluster)
    _check(L, ctx, rng)
