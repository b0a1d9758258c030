"""Appending a frame to the window copies its K, V and position rows and touches nothing else: frame sizes around the copy
kernel's blocks, both types and head dimensions, several appends in a row."""
from __future__ import annotations

import pytest
import torch

from paper_2601_04359_b200 import binding as pc

pytestmark = pytest.mark.gpu


# 64 fp32 rows of 2 x 64 are exactly two blocks of chunks for K and for V each; one token; ragged ends
@pytest.mark.parametrize("heads,d,dtype,frames", [((4, 2), 64, torch.float32, (64, 1, 63)), ((2, 1), 64, torch.bfloat16, (1, 1, 5)),
                                                  ((24, 8), 128, torch.bfloat16, (135, 1, 1008)), ((6, 6), 128, torch.float32, (257, 3))])
def test_append_copies_rows(heads, d, dtype, frames):
    total = sum(frames)
    ctx = pc.Context(heads[0], heads[1], d, pc.PC_BF16 if dtype == torch.bfloat16 else pc.PC_F32, 10000.0, (16, 16, 16), max(frames), total + 8)
    g = torch.Generator(device="cuda").manual_seed(total)
    rows = lambda n: torch.randn((n, heads[1], d), generator=g, device="cuda").to(dtype)
    pos = lambda n: torch.randint(0, 16, (n, 4), generator=g, dtype=torch.int32, device="cuda")
    mk = lambda n, x: pc.Segment(torch.full((n, heads[1], d), x, dtype=dtype, device="cuda"), torch.full((n, heads[1], d), x, dtype=dtype, device="cuda"),
                                 torch.full((n, 4), -3, dtype=torch.int32, device="cuda"), 0)
    a, b = mk(total + 8, 5.0), mk(total + 8, 5.0)
    win = pc.Window(ctx, len(frames) + 1, pc.PC_LINEAR, 0.0, total + 8, 0, pc.Segment.empty(), a, b)
    done = [pc.Segment(rows(n), rows(n), pos(n), n) for n in frames]
    for f in done:
        win.append(f)
    assert pc.pc_poll_status(ctx) == pc.PC_OK and win.state()[0].tolist() == list(frames)
    for have, name in ((a.k, "k"), (a.v, "v"), (a.pos, "pos")):
        assert torch.equal(have[:total], torch.cat([getattr(f, name) for f in done]))
    assert (a.k[total:] == 5.0).all() and (a.v[total:] == 5.0).all() and (a.pos[total:] == -3).all()
    assert (b.k == 5.0).all() and (b.pos == -3).all()
    win.close()
    ctx.close()
