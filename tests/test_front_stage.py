"""Scores, selection and pack of a small history in one launch (clusters of CTAs) against a kernel for each, bit for bit: the stage
marks of pc_set_timing keep the stages apart, so the same call on the same context gives both.  Frames around what a CTA scores at
once (32 keys), numbers of frames at which the clusters change, frames of unequal length and without tokens, and equal scores."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2601_04359_b200 import binding as pc

pytestmark = pytest.mark.gpu
BF, F32 = (24, 8, 128, torch.bfloat16), (4, 2, 64, torch.float32)

CASES = {
    "one_frame": (BF, [17], [5]),
    "two_tokens_a_cta": (BF, [9], [9]),
    "full_ctas": (BF, [256, 255], [100, 255]),
    "one_past": (BF, [257, 31], [64, 1]),
    "unequal": (BF, [3, 200, 0, 41, 1, 130], [1, 77, 0, 41, 0, 129]),
    "eleven_frames": (BF, [60] * 11, list(range(0, 55, 5))),
    "twelve_frames_two_a_cluster": (BF, [60] * 12, [7] * 12),
    "clusters_of_four": (BF, [120] * 17, [33] * 17),
    "frames_share_a_cta": (BF, [5, 9] * 48, [2, 9] * 48),
    "most_frames": (BF, [4] * 128, [1, 4] * 64),
    "too_many_frames": (BF, [4] * 129, [1] * 129),
    "rows_of_one_kb": ((16, 4, 128, torch.bfloat16), [330, 384], [50, 300]),
    "rows_of_four_kb": ((32, 16, 128, torch.bfloat16), [50, 64, 2], [25, 63, 1]),
    "six_heads": ((12, 6, 128, torch.bfloat16), [70, 8], [31, 2]),
    "fp32": (F32, [64] * 6, [32, 16, 8, 4, 2, 1]),
    "fp32_long": (F32, [300, 11], [20, 11]),
    "fp32_heads_of_128": ((3, 3, 128, torch.float32), [40, 100], [13, 50]),
    "bf16_heads_of_64": ((8, 4, 64, torch.bfloat16), [40, 100], [13, 50]),
    "nothing_kept": (BF, [30, 30], [0, 0]),
}


def _layer(heads, counts, n_q=37, seed=0, ties=True):
    hq, hk, d, dt = heads
    g = torch.Generator(device="cuda").manual_seed(seed)
    rand = lambda n, h: torch.randn(n, h, d, generator=g, device="cuda").to(dt)
    n = sum(counts)
    k = rand(n, hk)
    pos = torch.randint(4, 40, (n, 4), generator=g, device="cuda", dtype=torch.int32)
    if ties and n > 3:                                    # every third key is the one before it again, at the same place
        i = torch.arange(2, n, 3, device="cuda")
        k[i], pos[i] = k[i - 1], pos[i - 1]
    ctx = pc.Context(hq, hk, d, pc.PC_BF16 if dt == torch.bfloat16 else pc.PC_F32, 10000.0, (64, 64, 64), n_q, n + 8)
    anchors = pc.Segment(rand(5, hk), rand(5, hk), torch.randint(0, 40, (5, 4), generator=g, device="cuda", dtype=torch.int32), 5)
    cache = pc.Cache(anchors, pc.Segment(k, rand(n, hk), pos, n), np.array(counts, np.int32))
    q_pos = torch.randint(0, 40, (n_q, 4), generator=g, device="cuda", dtype=torch.int32)
    return ctx, cache, rand(n_q, hq), q_pos, g


def _step(ctx, cache, q, q_pos, quota, delta_t):
    n, total = cache.history.n_tokens, int(quota.sum())
    k = cache.history.k
    dst = pc.Cache(cache.anchors, pc.Segment(torch.full((total + 3,) + k.shape[1:], 5.0, dtype=k.dtype, device="cuda"),
                                             torch.full((total + 3,) + k.shape[1:], 5.0, dtype=k.dtype, device="cuda"),
                                             torch.full((total + 3, 4), -3, dtype=torch.int32, device="cuda"), 0), np.zeros(len(quota), np.int32))
    scores, sel = torch.full((n,), 7.0, device="cuda"), torch.full((total + 8,), -7, dtype=torch.int32, device="cuda")
    out, _, _, lse = pc.pc_frame_step(ctx, cache, quota, delta_t, dst, q, q_pos, scores=scores, sel_idx=sel, want_lse=True)
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    return [scores, sel, dst.history.k, dst.history.v, dst.history.pos, out, lse]


@pytest.mark.parametrize("case", list(CASES))
def test_one_launch_gives_the_bits_of_the_stages(case):
    heads, counts, quota = CASES[case]
    ctx, cache, q, q_pos, _ = _layer(heads, counts)
    quota = np.array(quota, np.int32)
    one = _step(ctx, cache, q, q_pos, quota, 3)
    pc.pc_set_timing(ctx, True)
    stages = _step(ctx, cache, q, q_pos, quota, 3)
    for a, b in zip(one, stages):
        assert torch.equal(a, b)
    pc.pc_set_timing(ctx, False)
    again = _step(ctx, cache, q, q_pos, quota, 3)         # the pooled query's accumulator was clear again
    assert all(torch.equal(a, b) for a, b in zip(one, again))
    ctx.close()


@pytest.mark.parametrize("counts,quota", [([60, 90, 31], [20, 5, 31]), ([300] * 2, [100, 7]), ([50] * 20, [9] * 20)])
def test_scores_and_selection_under_a_mask(counts, quota):
    ctx, cache, q, q_pos, g = _layer(BF, counts)
    quota = np.array(quota, np.int32)
    valid = (torch.rand(sum(counts), generator=g, device="cuda") < 0.5).to(torch.uint8)
    got = []
    for timing in (False, True):
        pc.pc_set_timing(ctx, timing)
        sel = torch.full((int(quota.sum()) + 4,), -7, dtype=torch.int32, device="cuda")
        scores, _ = pc.pc_score(ctx, cache, q, q_pos, quota, valid=valid, sel_idx=sel)
        assert pc.pc_poll_status(ctx) == pc.PC_OK
        got.append((scores.clone(), sel))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    assert bool((got[0][0][valid == 0] == -float("inf")).all())
    ctx.close()


def test_a_score_that_is_no_number_is_reported():
    ctx, cache, q, q_pos, _ = _layer(BF, [40, 40], ties=False)
    cache.history.k[50, 3, 7] = float("nan")
    pc.pc_score(ctx, cache, q, q_pos, np.array([5, 0], np.int32))
    assert pc.pc_poll_status(ctx) == pc.PC_OK             # not in a frame that is selected from
    pc.pc_score(ctx, cache, q, q_pos, np.array([5, 5], np.int32))
    assert pc.pc_poll_status(ctx) == pc.PC_ERR_INVALID_ARG
    ctx.close()


def test_keys_that_do_not_come():
    """The wait for the keys runs out: nothing is selected from what is not there, and the next call is whole again."""
    ctx, cache, q, q_pos, _ = _layer(BF, [60, 200, 90])
    quota = np.array([20, 50, 9], np.int32)
    good = _step(ctx, cache, q, q_pos, quota, 0)
    pc.pc_set_wait_limit_us(ctx, 2000)
    pc.pc_test_expect_extra_bytes(ctx, 16)
    sel = torch.full((int(quota.sum()) + 8,), -7, dtype=torch.int32, device="cuda")
    pc.pc_score(ctx, cache, q, q_pos, quota, sel_idx=sel)
    assert pc.pc_poll_status(ctx) == pc.PC_ERR_TIMEOUT
    assert bool((sel == -7).all())
    pc.pc_test_expect_extra_bytes(ctx, 0)
    pc.pc_set_wait_limit_us(ctx, 0)
    assert all(torch.equal(a, b) for a, b in zip(good, _step(ctx, cache, q, q_pos, quota, 0)))
    ctx.close()
