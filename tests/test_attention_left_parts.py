"""Items that two CTAs share and that are merged in the attention kernel, where that goes other than planned: a first part whose second
one does not come in time is left to the call's last CTA.  An odd number of query tiles (the second copy of one is dropped), a ragged last key
tile, boundaries reckoned in and not, more items than CTAs; against the oracle, and the same bits either way."""
from __future__ import annotations

from dataclasses import replace

import numpy as np
import pytest
import torch

import oracle
from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import workload as wl
from paper_2601_04359_b200.device import DeviceLayer, host, make_ctx

from .host_runtime import Case, _library, rt  # noqa: F401
from .test_randomized_shapes import abs_v, attention_within_bounds

# heads, grid of a frame, keys
MERGED = [((24, 8), (24, 42), 33 * 128), ((24, 8), (1, 1601), 4225), ((40, 8), (1, 1601), 1537), ((24, 8), (1, 1660), 1152), ((8, 8), (64, 92), 9 * 128 - 3)]


@pytest.mark.parametrize("heads,grid,n_keys", MERGED)
def test_merged_without_a_launch_of_its_own(rt, heads, grid, n_keys):
    rows = grid[0] * grid[1]
    c = Case(rt, heads=heads + (128,), n=1, total=1, anchors=1, max_q=rows, max_keys=n_keys)
    empty = lambda n, h: torch.empty(n, h, 128, dtype=torch.bfloat16)  # noqa: E731
    s = pc.Cache(pc.Segment(empty(n_keys, heads[1]), empty(n_keys, heads[1]), torch.empty(n_keys, 4, dtype=torch.int32), n_keys), pc.Segment.empty(), np.zeros(0, np.int32)).c()
    q, out, pos = empty(rows, heads[0]), empty(rows, heads[0]), torch.empty(rows, 4, dtype=torch.int32)
    rt.reset()
    assert rt.lib.pc_attend_frame(c.ctx.handle, pc.C.byref(s), None, pc._ptr(q), pc._ptr(pos), rows, pc._ptr(out), None, None) == pc.PC_OK
    assert [line.split()[1] for line in rt.log() if line.startswith("launch")] == ["k_rope_rows", "k_attend_tc"]


@pytest.mark.gpu
@pytest.mark.parametrize("heads,grid,n_keys", MERGED)
def test_left_parts_are_merged_by_the_last_cta(heads, grid, n_keys):
    hq, hkv = heads
    cfg = replace(wl.small_bf16(n_frames=1, grid=grid, n_text=1, seed=92), outliers=False, n_q_heads=hq, n_kv_heads=hkv)
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
    rows = np.array([(min(t * 128 + int(rng.integers(128)), cfg.n_q - 1), h) for t in range((cfg.n_q + 127) // 128) for h in range(hq)], np.int32)
    segs = [(L.hist_k, L.hist_v, L.hist_pos)]
    want, want_lse = oracle.attend(L.q, L.q_pos, segs, rows=rows, want_lse=True)
    got = host(out)[rows[:, 0], rows[:, 1]].astype(np.float64)
    assert attention_within_bounds(got, want, oracle.attend(L.q, L.q_pos, abs_v(segs), rows=rows))
    assert np.abs(host(lse)[rows[:, 0], rows[:, 1]] - want_lse).max() <= 2e-2

    again, lse2 = torch.zeros_like(out), torch.zeros_like(lse)
    attend = lambda: pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos, out=again, lse=lse2)  # noqa: E731
    for leave in (True, True, False, True):
        pc.pc_test_leave_parts(ctx, leave)
        again.zero_()
        lse2.zero_()
        attend()
        assert pc.pc_poll_status(ctx) == pc.PC_OK and torch.equal(again, out) and torch.equal(lse2, lse)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):                             # captured with everything left to the last CTA
        attend()
    for _ in range(2):
        again.zero_()
        g.replay()
        assert pc.pc_poll_status(ctx) == pc.PC_OK and torch.equal(again, out) and torch.equal(lse2, lse)
    del g
    ctx.close()


@pytest.mark.gpu
def test_a_cta_that_waits_for_an_sm_is_no_timeout():
    """Another stream's attention holds two SMs for longer than this call takes, so its last two CTAs start when others are done; the one in
    front of them has the first part of an item of which they have half.  The limit is a quarter of what that half takes and far
    above any wait of a CTA for its own copies and multiply-adds.  (A call whose limit is reached would say so and return: nothing hangs.)"""
    gen = torch.Generator(device="cuda").manual_seed(7)

    def layer(heads, n_q, n_keys):
        rand = lambda n: torch.randn(n, heads, 128, generator=gen, device="cuda").to(torch.bfloat16)  # noqa: E731
        ctx = pc.Context(heads, heads, 128, pc.PC_BF16, 10000.0, (64, 64, 64), n_q, n_keys)
        pos = lambda n: torch.randint(0, 64, (n, 4), generator=gen, device="cuda", dtype=torch.int32)  # noqa: E731
        cache = pc.Cache(pc.Segment(rand(n_keys), rand(n_keys), pos(n_keys), n_keys), pc.Segment.empty(), np.zeros(0, np.int32))
        pc.pc_attend_prepare(ctx, cache)
        q = rand(n_q)
        return ctx, cache, q, pos(n_q), torch.zeros_like(q)

    big = layer(8, 46 * 128, 96_000)                      # 184 items of 750 steps on 148 CTAs
    few = layer(2, 128, 400_000)                          # 2 items of 3,125 steps, one range each
    pc.pc_set_kv_splits(few[0], 1)
    attend = lambda x: pc.pc_attend_prepared(x[0], x[2], x[3], out=x[4])  # noqa: E731
    attend(few)
    attend(big)
    torch.cuda._sleep(1000)                               # a kernel's first launch may wait for what runs
    torch.cuda.synchronize()
    want = big[4].clone()
    big[4].zero_()
    pc.pc_set_wait_limit_us(big[0], 120)
    other = torch.cuda.Stream()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    end = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        attend(few)
        end.record()
    torch.cuda._sleep(100_000)                            # the other stream's kernels are on their SMs
    a.record()
    attend(big)
    b.record()
    torch.cuda.synchronize()
    assert a.elapsed_time(end) > 0.5 * a.elapsed_time(b)  # it was there while this call ran
    assert pc.pc_poll_status(big[0]) == pc.PC_OK and torch.equal(big[4], want)
    for x in (big, few):
        x[0].close()
