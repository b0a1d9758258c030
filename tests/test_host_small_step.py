"""The window step from host memory that goes up and home by a kernel each (small steps from pinned memory): its route, and that a
step that fails at whatever call leaves the window as it was."""
from __future__ import annotations

import ctypes as C

import pytest

from paper_2601_04359_b200 import binding as pc

from .host_runtime import PINNED, Case, _library, counts, rt  # noqa: F401


def launches(rt):
    return [line.split()[1] for line in rt.log() if line.startswith("launch")]


def state(win):
    c, t_shift, active = win.state()
    cache = pc.pc_cache()
    assert pc.load().pc_window_cache(win.handle, C.byref(cache)) == pc.PC_OK
    return c.tolist(), t_shift, active, cache.history.n_tokens, cache.history.k


@pytest.mark.parametrize("n", [36, 130])                  # scores, selection and pack in one launch with 36 tokens
@pytest.mark.parametrize("frames", [0, 1, 2, 4])          # fill, pack, pack, slide
def test_small_step_that_fails_leaves_the_window(rt, frames, n):
    def case():
        c = Case(rt, n=n, total=100 if n == 36 else 200, window=3).pin()
        win = c.make()
        for _ in range(frames):
            c.step_host(win)
        return c, win

    c, probe = case()
    rt.reset()
    c.step_host(probe)
    assert launches(rt)[0] == launches(rt)[-1] == "k_move" and not any(line.startswith("memcpy") for line in rt.log())
    if frames >= 4:
        assert "k_front" in launches(rt)
    want = state(probe)[:4]
    for name in {line.split()[0] for line in rt.log()} - {"synchronize"}:
        c, win = case()
        for at in range(99):                              # until there is no call left to fail
            before = state(win)
            rt.reset()
            rt.fail(name, at)
            try:
                c.step_host(win)
                break
            except pc.PackCacheError as e:
                assert e.status == pc.PC_ERR_CUDA and state(win) == before
                assert sorted(rt.log()[-2:]) == ["synchronize main", "synchronize side"]
        assert at > 0 and state(win)[:4] == want          # and the same step still works


@pytest.mark.parametrize("which", ["q", "q_pos", "k", "v", "pos", "out"])
def test_memory_that_is_pinned_at_both_ends_only_goes_by_copies(rt, which):
    """Two registered ranges with pageable memory in between: a kernel that read it would fault."""
    c = Case(rt, n=130, total=200).pin()
    win = c.make()
    t = {"q": c.q, "q_pos": c.q_pos, "out": c.out, "k": c.frame.k, "v": c.frame.v, "pos": c.frame.pos}[which]
    rt.memory(t[:40], t[90:], kind=PINNED)
    rt.reset()
    c.step_host(win)
    copies = sum(line.startswith("memcpy") for line in rt.log())
    # positions by copies as well if they are what is not pinned in whole
    assert copies == (5 if which in ("q_pos", "pos") else 4) and launches(rt)[-1] != "k_move"
    rt.memory(t, kind=PINNED)
    rt.reset()
    c.step_host(win)
    assert launches(rt)[0] == launches(rt)[-1] == "k_move" and not any(line.startswith("memcpy") for line in rt.log())
