"""The rotary pre-pass at every width of key row that has a kernel of its own (chunks per lane 1, 2, 3, 4, 5, 7, 11, 13) and at rows of
several slices, against the CUDA-core kernel, which rotates on its way into shared memory: two bf16 roundings of the rotated
operands and one of the probabilities apart, which move a result by at most 2^-6 of sum p |v| (the bound of the random-shape tests),
and a rounding of the result on either side."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2601_04359_b200 import binding as pc

from .test_gpu_parity import bf16_ulp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_kv,group", [(2, 1), (2, 3), (4, 2), (6, 1), (8, 3), (10, 2), (12, 1), (14, 1), (16, 2), (18, 1), (20, 1), (22, 1), (26, 1), (32, 1)])
def test_rotated_rows(n_kv, group):
    n, n_q = 131, 9
    g = torch.Generator(device="cuda").manual_seed(n_kv)
    rows = lambda m, h: torch.randn((m, h, 128), generator=g, device="cuda").bfloat16()
    pos = lambda m: torch.randint(0, 32, (m, 4), generator=g, dtype=torch.int32, device="cuda")
    ctx = pc.Context(n_kv * group, n_kv, 128, pc.PC_BF16, 10000.0, (32, 32, 32), n_q, 2 * n)
    cache = pc.Cache(pc.Segment(rows(5, n_kv), rows(5, n_kv), pos(5), 5), pc.Segment(rows(n, n_kv), rows(n, n_kv), pos(n), n), np.array([n], np.int32))
    q, q_pos = rows(n_q, n_kv * group), pos(n_q)
    got = pc.pc_attend_frame(ctx, cache, None, q, q_pos)
    pc.pc_attend_prepare(ctx, cache)                                   # keys and queries in launches of their own: the same bits
    assert torch.equal(pc.pc_attend_prepared(ctx, q, q_pos), got)
    pc.pc_set_attend_impl(ctx, 1)
    want = pc.pc_attend_frame(ctx, cache, None, q, q_pos).float().cpu().numpy()
    for s in (cache.anchors, cache.history):
        s.v.abs_()
    mean_abs = pc.pc_attend_frame(ctx, cache, None, q, q_pos).float().cpu().numpy()
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    assert (np.abs(got.float().cpu().numpy() - want) <= 2 * bf16_ulp(want) + 2.0 ** -6 * mean_abs + 1e-3).all()
    ctx.close()
