"""Host-side behaviour of the library's calls, over a CUDA runtime that runs nothing."""
from __future__ import annotations

import ctypes as C

import numpy as np
import pytest
import torch

from paper_2601_04359_b200 import binding as pc

from .host_runtime import CALLBACK, DEVICE, PINNED, Case, _library, counts, rt  # noqa: F401


def test_window_belongs_to_the_device_of_its_context(rt):
    c = Case(rt)                                          # the context lives on device 0
    rt.device(1)
    win = c.make()
    dev = C.c_int(-1)
    rt.lib.cudaGetDevice(C.byref(dev))
    assert dev.value == 1                                 # creating the window leaves the caller's device as it was
    rt.device(0)
    for n in range(1, 4):                                 # fill, then pack
        c.step_host(win)
        assert len(counts(win)) == n


def _refused(win, case, log, **kw):
    before, (_, _, active) = counts(win), win.state()
    case.rt.reset()
    with pytest.raises(pc.PackCacheError) as e:
        case.step_host(win, **kw)
    assert counts(win) == before and win.state()[2] == active
    if not log:
        assert case.rt.log() == []                        # nothing was enqueued
    return e.value.status


def test_host_step_checks_before_it_enqueues(rt):
    c = Case(rt)
    win = c.make()
    skew = torch.zeros(c.ws["q"].numel() + 8, dtype=torch.bfloat16)[1:1 + c.ws["q"].numel()].view_as(c.ws["q"])
    for f in range(3):                                    # fill, fill to the brim, pack
        for name in ("q", "out"):
            assert _refused(win, c, False, **{name: skew}) == pc.PC_ERR_INVALID_ARG
        c.step_host(win)
        assert len(counts(win)) == f + 1
    few = Case(rt, max_keys=200)                          # 37 anchors and 130 tokens fit, two frames (packed to 200 tokens) do not
    win = few.make()
    few.step_host(win)
    assert _refused(win, few, False) == pc.PC_ERR_CAPACITY
    odd = Case(rt, heads=(10, 5, 128))                    # key rows of 1,280 bytes: attention takes them, scoring does not
    win = odd.make()
    odd.step_host(win)
    assert _refused(win, odd, False) == pc.PC_ERR_UNSUPPORTED


@pytest.mark.parametrize("frames", [0, 1, 2])
def test_host_step_that_fails_leaves_the_window_and_nothing_in_flight(rt, frames):
    c = Case(rt)
    win = c.make()
    for _ in range(frames):
        c.step_host(win)
    rt.reset()
    probe = c.make()
    for _ in range(frames + 1):
        rt.reset()
        c.step_host(probe)
    calls = [line.split()[0] for line in rt.log()]
    for name in ("memcpy", "record", "wait", "launch"):
        for at in range(calls.count(name)):
            rt.reset()
            rt.fail(name, at)
            before, active = counts(win), win.state()[2]
            with pytest.raises(pc.PackCacheError) as e:
                c.step_host(win)
            assert e.value.status == pc.PC_ERR_CUDA
            assert counts(win) == before and win.state()[2] == active
            assert sorted(rt.log()[-2:]) == ["synchronize main", "synchronize side"]
    rt.reset()
    c.frame.k.fill_(3.0)
    c.step_host(win)                                      # and the same step still works
    assert len(counts(win)) == frames + 1
    assert counts(win) == counts(probe)


def test_two_threads_scoring_rows_of_different_width(rt):
    """The query pass of 32 heads x 128 takes 64 KB of shared memory a block, that of 40 heads 60 KB, in the same kernel.  The
    second thread's first call comes while the first one's is between raising the limit and launching."""
    cases = [Case(rt, heads=(hq, 8, 128), n=8) for hq in (32, 40)]
    cache, budget = pc.Cache(pc.Segment.empty(), cases[0].frame, np.array([8], np.int32)), (C.c_int32 * 1)(4)
    scores, sel = torch.zeros(8), torch.zeros(8, dtype=torch.int32)
    status = []

    def score(c):
        s = cache.c()
        status.append(rt.lib.pc_score(c.ctx.handle, C.byref(s), pc._ptr(c.q), pc._ptr(c.q_pos), 8, budget, None, None, pc._ptr(scores), pc._ptr(sel), None))

    other = CALLBACK(lambda: score(cases[1]))
    rt.lib.rt_on_attribute(other)
    score(cases[0])
    score(cases[1])
    score(cases[0])
    assert status == [pc.PC_OK] * 4


@pytest.mark.parametrize("n_kv,status", [(4, pc.PC_OK), (5, pc.PC_ERR_UNSUPPORTED), (6, pc.PC_OK), (7, pc.PC_ERR_UNSUPPORTED), (8, pc.PC_OK)])
def test_static_scoring_takes_the_row_widths_that_scoring_takes(rt, n_kv, status):
    """fp32 key rows of n_kv x 512 bytes: 2,560 and 3,584 are refused with nothing enqueued."""
    desc = pc.pc_layer_desc(n_kv, n_kv, 128, pc.PC_F32, 10000.0, (C.c_int32 * 3)(64, 64, 64), 0, 0)
    k, pos, out, word = torch.zeros(8, n_kv, 128), torch.zeros(8, 4, dtype=torch.int32), torch.zeros(8), torch.zeros(2, dtype=torch.int32)
    got = rt.lib.pc_score_tokens_static(C.byref(desc), pc._ptr(k), pc._ptr(pos), 8, pc._ptr(k), pc._ptr(pos), 8, None, pc._ptr(out), pc._ptr(word), None)
    assert got == status
    assert [line.split()[1] for line in rt.log()] == (["k_rope_table", "k_qprep", "k_score"] if status == pc.PC_OK else [])


def test_scratch_of_a_context_per_key(rt):
    """A key costs its rotated row (8 x 128 bf16) and, for the attention mass, one fp32 sum per KV head and column half."""
    size = []
    for keys in (50_000, 250_000):
        rt.reset()
        pc.Context(24, 8, 128, pc.PC_BF16, 10000.0, (64, 64, 64), 1008, keys).close()
        size.append(sum(int(line.split()[1]) for line in rt.log() if line.startswith("malloc")))
    assert (size[1] - size[0]) / 200_000 <= 8 * 128 * 2 + 8 * 2 * 4 + 1


def test_stage_times_of_a_step_in_parts(rt):
    """520 rows of 24 / 8 heads leave in two parts: the stages cover both, and the rotary pre-pass ahead of them."""
    c = Case(rt, n=520, total=600)
    win = c.make()
    pc.pc_set_timing(c.ctx, True)
    for f in range(2):                                    # fill: everything is rotated; pack: query pass, scores, selection, pack, the anchors' keys
        rt.reset()
        c.step_host(win)
        log = [line.split()[1] for line in rt.log() if line.startswith("launch")]
        assert log.count("k_attend_tc") == 2 and log.count("k_rope_rows") == 1
        t = pc.pc_get_timing(c.ctx)
        assert t["rope"] == 1 and t["rope"] + t["attend"] + max(t["combine"], 0) == len(log) - (4 if f else 0)
        assert t["attend"] == len(log) - 1 - log[::-1].index("k_attend_tc") - log.index("k_rope_rows")


@pytest.mark.parametrize("heads,rows", [((24, 8), 385), ((32, 8), 385), ((24, 12), 385), ((32, 16), 385), ((16, 4), 641), ((8, 8), 1153),
                                        ((64, 8), 129), ((32, 32), 129), ((24, 24), 129)])
def test_rows_from_which_a_step_runs_in_parts(rt, heads, rows):
    """The numbers that the header states, for 148 SMs."""
    for n, parts in ((rows - 1, 1), (rows, 2)):
        c = Case(rt, heads=heads + (128,), n=n, total=n)
        rt.reset()
        c.step_host(c.make())
        assert sum("k_attend_tc" in line for line in rt.log()) == parts


@pytest.mark.parametrize("kind,device,route", [(DEVICE, 0, ["launch k_append main"]), (DEVICE, 1, ["memcpy main"] * 3), (PINNED, 0, ["memcpy main"] * 3),
                                               (0, 0, ["memcpy main"] * 3)])
@pytest.mark.parametrize("which", ["k", "v", "pos"])
def test_append_reads_only_its_own_device_with_a_kernel(rt, kind, device, route, which):
    """A frame on another GPU, in pinned memory, or in memory the driver does not know goes by the runtime's copies, which
    reach it or refuse it; a kernel would fault."""
    c = Case(rt)
    win = c.make()
    c.frame.k.normal_()
    rt.memory(getattr(c.frame, which), kind=kind, device=device)
    rt.reset()
    f = c.frame.c()
    assert rt.lib.pc_window_append(win.handle, C.byref(f), None) == pc.PC_OK
    assert rt.log() == route and counts(win) == [c.n]
    if len(route) == 3:
        assert torch.equal(c.bufs[0].k[:c.n], c.frame.k)


@pytest.mark.parametrize("heads,rows,keys,blocks", [((24, 8), 1008, 48384, 144), ((24, 8), 1008, 9200, 144), ((8, 8), 1008, 48000, 144),
                                                    ((16, 16), 1008, 30000, 148), ((64, 8), 1008, 24000, 148), ((8, 8), 4032, 24000, 148),
                                                    ((24, 8), 4032, 9200, 148)])
def test_attention_gives_up_sms_only_for_shared_streams(rt, heads, rows, keys, blocks):
    """144 CTAs where a KV head's CTAs then run through the same keys two or more at a time, each over less than an item; every
    other shape keeps a CTA on each of the 148 SMs."""
    c = Case(rt, heads=(heads[0], heads[1], 128), n=1, total=1, anchors=1, max_q=rows, max_keys=keys)
    empty = lambda n: pc.Segment(torch.empty(n, heads[1], 128, dtype=torch.bfloat16), torch.empty(n, heads[1], 128, dtype=torch.bfloat16),
                                 torch.empty(n, 4, dtype=torch.int32), n)
    q, out = (torch.empty(rows, heads[0], 128, dtype=torch.bfloat16) for _ in range(2))
    s = pc.Cache(empty(keys), pc.Segment.empty(), np.zeros(0, np.int32)).c()
    pos = torch.empty(rows, 4, dtype=torch.int32)
    assert rt.lib.pc_attend_frame(c.ctx.handle, C.byref(s), None, pc._ptr(q), pc._ptr(pos), rows, pc._ptr(out), None, None) == pc.PC_OK
    assert rt.lib.rt_blocks(b"k_attend_tc") == blocks


def test_attention_is_not_launched_with_fewer_registers_than_its_warps_share_out(rt):
    """Its softmax warps ask for registers that the block must have been launched with, and wait for them without a limit."""
    rt.device(2)                                          # a device on which no other test has launched it
    c = Case(rt)
    rt.memory(c.q, c.q_pos, c.out, device=2)
    cache = pc.Cache(c.anchors, c.frame, np.array([c.n], np.int32)).c()
    attend = lambda: rt.lib.pc_attend_frame(c.ctx.handle, C.byref(cache), None, pc._ptr(c.q), pc._ptr(c.q_pos), c.n, pc._ptr(c.out), None, None)  # noqa: E731
    launched = lambda: [line for line in rt.log() if line.startswith("launch k_attend")]  # noqa: E731
    rt.lib.rt_registers(160)
    assert attend() == pc.PC_ERR_CUDA and not launched()
    rt.lib.rt_registers(168)
    assert attend() == pc.PC_OK and len(launched()) == 1


def test_a_merge_is_reckoned_as_what_it_takes(rt):
    """40 items of four key tiles: two ranges each (80 CTAs) save two steps and cost a merge, which is as long; one range, no merge."""
    c = Case(rt, n=300, anchors=304)
    one = pc.Segment(c.frame.k, c.frame.v, c.frame.pos, 1)
    cache = pc.Cache(c.anchors, one, np.array([1], np.int32)).c()
    rt.lib.rt_blocks.argtypes = [C.c_char_p]
    assert rt.lib.pc_attend_frame(c.ctx.handle, C.byref(cache), None, pc._ptr(c.q), pc._ptr(c.q_pos), c.n, pc._ptr(c.out), None, None) == pc.PC_OK
    assert rt.lib.rt_blocks(b"k_attend_tc") == 40
    assert not [line for line in rt.log() if line.startswith("launch k_combine")]
