"""Items that two CTAs share: the one with the first part adds the second to it at the end of its run.  Whole frames whose runs cross
items, two fixed key ranges (which end together and are merged by a kernel of their own), an odd number of query tiles, rows past the last;
against the oracle, and the same bits again from call to call, from a captured graph, and after a call that gave up."""
from __future__ import annotations

from dataclasses import replace

import numpy as np
import pytest
import torch

import oracle
from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import workload as wl
from paper_2601_04359_b200.device import DeviceLayer, host, make_ctx

from .test_randomized_shapes import abs_v, attention_within_bounds

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,grid,n_keys,splits", [((24, 8), (24, 42), 11 * 128 - 7, 0), ((24, 8), (24, 42), 33 * 128, 0), ((40, 8), (20, 30), 12 * 128 + 1, 0),
                                                      ((8, 8), (1, 100), 6 * 128, 2), ((24, 8), (9, 15), 3 * 128 - 50, 2), ((5, 5), (3, 131), 2 * 128, 2)])
def test_two_parts(heads, grid, n_keys, splits):
    hq, hkv = heads
    if (hkv * 128) % 256:
        hq, hkv = hq + 1, hkv + 1
    cfg = replace(wl.small_bf16(n_frames=1, grid=grid, n_text=1, seed=91), outliers=False, n_q_heads=hq, n_kv_heads=hkv)
    L = wl.make_layer(cfg)
    rng = np.random.default_rng(n_keys)
    L.hist_k, L.hist_v = (wl.round_bf16(rng.standard_normal((n_keys, hkv, 128)).astype(np.float32)) for _ in range(2))
    L.hist_pos = np.stack([np.arange(n_keys) % 10, np.arange(n_keys) % cfg.max_pos[1], np.arange(n_keys) % cfg.max_pos[2], np.arange(n_keys)], axis=1).astype(np.int32)
    L.frame_count = np.array([n_keys], np.int32)
    L.anchor_k, L.anchor_v, L.anchor_pos = L.anchor_k[:0], L.anchor_v[:0], L.anchor_pos[:0]
    D = DeviceLayer(L)
    ctx = make_ctx(cfg, max_keys=n_keys)
    pc.pc_set_kv_splits(ctx, splits)
    out, lse = pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos, want_lse=True)
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    rows = np.array([(min(t * 128 + int(rng.integers(128)), cfg.n_q - 1), h) for t in range((cfg.n_q + 127) // 128) for h in range(hq) for _ in range(2)], np.int32)
    segs = [(L.hist_k, L.hist_v, L.hist_pos)]
    want, want_lse = oracle.attend(L.q, L.q_pos, segs, rows=rows, want_lse=True)
    got = host(out)[rows[:, 0], rows[:, 1]].astype(np.float64)
    assert attention_within_bounds(got, want, oracle.attend(L.q, L.q_pos, abs_v(segs), rows=rows))
    assert np.abs(host(lse)[rows[:, 0], rows[:, 1]] - want_lse).max() <= 2e-2

    again, lse2 = torch.zeros_like(out), torch.zeros_like(lse)
    attend = lambda: pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos, out=again, lse=lse2)  # noqa: E731
    same = lambda: pc.pc_poll_status(ctx) == pc.PC_OK and torch.equal(again, out) and torch.equal(lse2, lse)  # noqa: E731
    for _ in range(3):
        again.zero_()
        attend()
        assert same()
    pc.pc_set_wait_limit_us(ctx, 2000)
    pc.pc_test_expect_extra_bytes(ctx, 16)
    attend()
    assert pc.pc_poll_status(ctx) == pc.PC_ERR_TIMEOUT
    pc.pc_test_expect_extra_bytes(ctx, 0)
    pc.pc_set_wait_limit_us(ctx, 0)
    again.zero_()
    attend()
    assert same()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        attend()
    for _ in range(3):
        again.zero_()
        lse2.zero_()
        g.replay()
        assert same()
    del g
    ctx.close()
