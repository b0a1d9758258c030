"""A bounded device-side wait that runs out, on purpose and in the permitted form.

Every wait of the library's kernels has a limit; when it runs out the kernel records PC_ERR_TIMEOUT, gives up the work
that depended on the wait, lets its copies land, frees what it holds and returns, and the context stays usable.  Here
the limit is set to two milliseconds and the attention kernel's first barrier is told by the host to expect sixteen
bytes more than its copies will ever deliver, so the wait on it cannot be satisfied: nothing traps, nothing spins
without a limit, no address is bad.  The next ordinary call on the same context must work and match the oracle."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import workload as wl
from paper_2601_04359_b200.device import DeviceLayer, host, make_ctx

from .test_gpu_parity import check_bf16_attention

pytestmark = pytest.mark.gpu


def test_a_wait_that_runs_out_is_reported_and_the_context_survives():
    cfg = wl.small_bf16(n_frames=2, grid=(8, 9), seed=60)
    L = wl.make_layer(cfg)
    D = DeviceLayer(L)
    ctx = make_ctx(cfg)
    good = pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos).clone()
    assert pc.pc_poll_status(ctx) == pc.PC_OK

    pc.pc_set_wait_limit_us(ctx, 2000)
    pc.pc_test_expect_extra_bytes(ctx, 16)
    pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos)          # every CTA's first wait runs out after 2 ms
    assert pc.pc_poll_status(ctx) == pc.PC_ERR_TIMEOUT
    assert pc.pc_poll_status(ctx) == pc.PC_OK                      # polling cleared the word

    pc.pc_test_expect_extra_bytes(ctx, 0)
    pc.pc_set_wait_limit_us(ctx, 0)
    again = pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos)
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    assert (again.view(dtype=good.dtype) == good).all()
    want = oracle.attend(L.q, L.q_pos, [(L.anchor_k, L.anchor_v, L.anchor_pos), (L.hist_k, L.hist_v, L.hist_pos)], cfg.rope_base)
    check_bf16_attention(host(again).astype(np.float64), want)
    ctx.close()


@pytest.mark.parametrize("n_frames,grid", [(2, (8, 9)), (9, (24, 42))])        # one group a warp, and a ring that goes round
def test_a_scoring_wait_that_runs_out(n_frames, grid):
    """The scoring kernel gives up, its last block still clears the pooled query's accumulator and ticket, and the next
    call's scores are the ones of a fresh context."""
    cfg = wl.small_bf16(n_frames=n_frames, grid=grid, seed=61)
    D = DeviceLayer(wl.make_layer(cfg))
    ctx = make_ctx(cfg)
    budget = np.full(n_frames, 7, np.int32)
    good, good_sel = pc.pc_score(ctx, D.cache, D.q, D.q_pos, budget)
    assert pc.pc_poll_status(ctx) == pc.PC_OK

    pc.pc_set_wait_limit_us(ctx, 2000)
    pc.pc_test_expect_extra_bytes(ctx, 16)
    pc.pc_score(ctx, D.cache, D.q, D.q_pos, budget)
    assert pc.pc_poll_status(ctx) == pc.PC_ERR_TIMEOUT
    assert pc.pc_poll_status(ctx) == pc.PC_OK

    pc.pc_test_expect_extra_bytes(ctx, 0)
    pc.pc_set_wait_limit_us(ctx, 0)
    again, again_sel = pc.pc_score(ctx, D.cache, D.q, D.q_pos, budget)
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    assert torch.equal(again, good) and torch.equal(again_sel, good_sel)
    ctx.close()


def test_a_mass_wait_that_runs_out():
    cfg = wl.small_bf16(n_frames=2, grid=(8, 9), seed=62)
    D = DeviceLayer(wl.make_layer(cfg))
    ctx = make_ctx(cfg)
    n_keys = cfg.n_anchor + cfg.n_src
    _, lse = pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos, want_lse=True)
    good = pc.pc_attend_mass(ctx, lse, n_keys)
    assert pc.pc_poll_status(ctx) == pc.PC_OK

    pc.pc_set_wait_limit_us(ctx, 2000)
    pc.pc_test_expect_extra_bytes(ctx, 16)
    pc.pc_attend_mass(ctx, lse, n_keys)
    assert pc.pc_poll_status(ctx) == pc.PC_ERR_TIMEOUT

    pc.pc_test_expect_extra_bytes(ctx, 0)
    pc.pc_set_wait_limit_us(ctx, 0)
    again = pc.pc_attend_mass(ctx, lse, n_keys)
    assert pc.pc_poll_status(ctx) == pc.PC_OK and torch.equal(again, good)
    ctx.close()


def _calls(ctx, D, cfg):
    budget = np.full(cfg.n_frames, 7, np.int32)
    n_keys = cfg.n_anchor + cfg.n_src
    _, lse = pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos, want_lse=True)
    calls = {"attend": lambda: pc.pc_attend_frame(ctx, D.cache, None, D.q, D.q_pos),
             "mass": lambda: pc.pc_attend_mass(ctx, lse, n_keys),
             "score": lambda: pc.pc_score(ctx, D.cache, D.q, D.q_pos, budget)}
    for call in calls.values():
        call()
    assert pc.pc_poll_status(ctx) == pc.PC_OK
    return calls


def _timed_out_ms(ctx, call, limit_us):
    pc.pc_set_wait_limit_us(ctx, limit_us)
    pc.pc_test_expect_extra_bytes(ctx, 16)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    call()
    b.record()
    assert pc.pc_poll_status(ctx) == pc.PC_ERR_TIMEOUT
    pc.pc_test_expect_extra_bytes(ctx, 0)
    pc.pc_set_wait_limit_us(ctx, 0)
    return a.elapsed_time(b)


def test_copies_get_time_to_land_whoever_gives_up():
    """A run of one step or two: the warp that issues the copies is done before another one gives up, and the copies still get
    their two milliseconds."""
    cfg = wl.small_bf16(n_frames=2, grid=(8, 9), seed=63)
    D = DeviceLayer(wl.make_layer(cfg))
    ctx = make_ctx(cfg)
    for name, call in _calls(ctx, D, cfg).items():
        ms = _timed_out_ms(ctx, call, 2000)
        assert ms >= 2 + 2, f"{name}: {ms:.2f} ms"
    ctx.close()


@pytest.mark.parametrize("limit_us", [200, 2000])
def test_a_wait_gives_up_when_its_limit_is_reached(limit_us):
    """A call whose first wait runs out takes the limit, the time that copies in flight get to land (2 ms) and a few questions of
    4 to 10 us each, and no more: 3 ms are left for those and the launches around the kernel."""
    cfg = wl.small_bf16(n_frames=2, grid=(8, 9), seed=64)
    D = DeviceLayer(wl.make_layer(cfg))
    ctx = make_ctx(cfg)
    for name, call in _calls(ctx, D, cfg).items():
        ms = min(_timed_out_ms(ctx, call, limit_us) for _ in range(3))      # a host held up between the launches counts as well
        assert ms <= limit_us / 1000 + 5, f"{name}: {ms:.2f} ms"
    ctx.close()
