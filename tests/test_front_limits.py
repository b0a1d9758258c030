"""Where the launch for small histories begins and ends: which kernels a step and a scoring call enqueue on both sides of each limit, and the
same bits on both sides of it."""
from __future__ import annotations

import ctypes as C

import numpy as np
import pytest
import torch

from paper_2601_04359_b200 import binding as pc

from .host_runtime import _library, rt  # noqa: F401
from .test_front_stage import _layer, _step

BF, F32 = torch.bfloat16, torch.float32

# heads, type, frames, most tokens of a frame: 36 of a CTA's 2 KB rows, 40 of 1.5 KB, 48 of 1 KB; 32 in clusters of four (40 and 48 of narrow bf16 rows)
STEP = [((24, 8, 128), BF, 1, 288), ((24, 8, 128), BF, 11, 288), ((24, 8, 128), BF, 12, 128), ((12, 6, 128), BF, 5, 320), ((12, 6, 128), BF, 16, 160),
        ((16, 4, 128), BF, 5, 384), ((16, 4, 128), BF, 32, 192), ((4, 2, 64), F32, 5, 384), ((4, 2, 64), F32, 12, 128), ((8, 4, 64), F32, 24, 128)]
SCORE = [((24, 8, 128), BF, 1, 256), ((24, 8, 128), BF, 2, 288), ((16, 4, 128), BF, 1, 256), ((32, 16, 128), BF, 5, 256)]


def _kernels(rt, heads, dt, counts, pack):
    hq, hk, d = heads
    n, n_q = sum(counts), 8
    ctx = pc.Context(hq, hk, d, pc.PC_BF16 if dt == BF else pc.PC_F32, 10000.0, (64, 64, 64), n_q, n + 8)
    rt.open.append(ctx)
    z = lambda m, h: torch.zeros(m, h, d, dtype=dt)  # noqa: E731
    pos = torch.zeros(n, 4, dtype=torch.int32)
    src = pc.Cache(pc.Segment.empty(), pc.Segment(z(n, hk), z(n, hk), pos, n), np.array(counts, np.int32))
    budget = (C.c_int32 * len(counts))(*[(c + 1) // 2 for c in counts])
    total = sum(budget)
    q, q_pos, scores, sel = z(n_q, hq), torch.zeros(n_q, 4, dtype=torch.int32), torch.zeros(n), torch.zeros(total, dtype=torch.int32)
    c_src = src.c()
    rt.reset()
    if pack:
        dst = pc.Cache(pc.Segment.empty(), pc.Segment(z(total, hk), z(total, hk), torch.zeros(total, 4, dtype=torch.int32), total), np.zeros(len(counts), np.int32))
        out, c_dst = torch.zeros_like(q), dst.c()
        assert pc.load().pc_frame_step(ctx.handle, C.byref(c_src), budget, 0, C.byref(c_dst), pc._ptr(q), pc._ptr(q_pos), n_q, pc._ptr(scores), pc._ptr(sel),
                                    pc._ptr(out), None, None) == pc.PC_OK
    else:
        assert pc.load().pc_score(ctx.handle, C.byref(c_src), pc._ptr(q), pc._ptr(q_pos), n_q, budget, None, None, pc._ptr(scores), pc._ptr(sel), None) == pc.PC_OK
    return [line.split()[1] for line in rt.log() if line.startswith("launch")]


@pytest.mark.parametrize("pack,case", [(True, c) for c in STEP] + [(False, c) for c in SCORE])
def test_which_kernels_a_call_enqueues(rt, pack, case):
    heads, dt, frames, most = case
    ctas = 8 if frames <= 11 else 4
    inside = _kernels(rt, heads, dt, [most] + [most - 1] * (frames - 1), pack)
    assert inside[:2] == ["k_qprep", "k_front"]
    assert (inside[2].startswith("k_attend") if pack else len(inside) == 2)
    beyond = _kernels(rt, heads, dt, [most + 1] + [most - 1] * (frames - 1), pack)
    assert "k_front" not in beyond and beyond[:2] == ["k_qprep", "k_score"] and most % ctas == 0


def test_which_kernels_few_tokens_of_many_frames_enqueue(rt):
    assert "k_front" in _kernels(rt, (4, 2, 64), F32, [64] * 16, True)
    assert "k_front" not in _kernels(rt, (4, 2, 64), F32, [64] * 17, True)      # fp32 rows of 512 bytes: sixteen frames
    assert "k_front" in _kernels(rt, (24, 8, 128), BF, [30] * 128, True)
    assert "k_front" not in _kernels(rt, (24, 8, 128), BF, [30] * 129, True)
    assert "k_front" not in _kernels(rt, (24, 8, 128), BF, [1008] * 47, True)


@pytest.mark.gpu
@pytest.mark.parametrize("past", [0, 1])
@pytest.mark.parametrize("heads,dt,frames,most", STEP)
def test_the_same_bits_at_the_limits(heads, dt, frames, most, past):
    counts = [most + past] + [most - 1] * (frames - 1)
    ctx, cache, q, q_pos, _ = _layer(heads + (dt,), counts)
    quota = np.array([max(1, c // 3) for c in counts], np.int32)
    one = _step(ctx, cache, q, q_pos, quota, 2)
    pc.pc_set_timing(ctx, True)
    stages = _step(ctx, cache, q, q_pos, quota, 2)
    assert all(torch.equal(a, b) for a, b in zip(one, stages))
    ctx.close()
