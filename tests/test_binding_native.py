"""The binding's native side, without a GPU: host arrays of any integer kind, tensors that are not contiguous, a closed
context."""
from __future__ import annotations

import importlib.machinery

import numpy as np
import pytest
import torch

from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import build


@pytest.mark.parametrize("make", [list, tuple, lambda a: np.array(a, np.int64), lambda a: np.array(a, np.int32),
                                  lambda a: np.array(a, np.int32).repeat(2)[::2], lambda a: torch.tensor(a, dtype=torch.int32),
                                  lambda a: np.array(a, np.int32)[:, None]])
def test_host_arrays_of_any_integer_kind(make):
    avail = [40, 7, 100, 0, 64]
    want = pc.pc_plan_budget(pc.PC_LINEAR, 0.0, 90, 0, np.array(avail, np.int32))
    got = pc.pc_plan_budget(pc.PC_LINEAR, 0, np.int64(90), np.int32(0), make(avail))
    assert got.dtype == np.int32 and got.tolist() == want.tolist() and want.sum() == 90


def _segment(n):
    return pc.Segment(torch.zeros(n, 2, 8), torch.zeros(n, 2, 8), torch.zeros(n, 4, dtype=torch.int32), n)


class _Closed:
    handle = None


def test_errors_reach_the_caller():
    q, q_pos = torch.zeros(4, 2, 8), torch.zeros(4, 4, dtype=torch.int32)
    cache = pc.Cache(pc.Segment.empty(), _segment(6), [2, 4])
    with pytest.raises(pc.PackCacheError) as e:                        # the library refuses a null context before it reads anything
        pc.pc_attend_frame(_Closed, cache, None, q, q_pos, stream=0)
    assert e.value.status == pc.PC_ERR_INVALID_ARG
    with pytest.raises(AssertionError, match="contiguous"):
        pc.pc_attend_frame(_Closed, cache, None, q.transpose(0, 1), q_pos, out=q, stream=0)
    with pytest.raises(ValueError):
        pc.pc_compact(_Closed, cache, q_pos, ["x"], 0, cache, stream=0)
    assert cache.history.n_tokens == 6                                 # a refused call leaves the destination's count alone


def test_a_budget_shorter_than_the_frames_is_refused():
    q, q_pos = torch.zeros(4, 2, 8), torch.zeros(4, 4, dtype=torch.int32)
    cache, sel = pc.Cache(pc.Segment.empty(), _segment(6), [2, 4]), torch.zeros(6, dtype=torch.int32)
    calls = [lambda b: pc.pc_score(_Closed, cache, q, q_pos, b, scores=q, sel_idx=sel, stream=0),
             lambda b: pc.pc_compact(_Closed, cache, sel, b, 0, cache, stream=0),
             lambda b: pc.pc_frame_step(_Closed, cache, b, 0, cache, q, q_pos, scores=q, sel_idx=sel, out=q, stream=0)]
    for call in calls:
        with pytest.raises(ValueError, match="budget has 1 entries, 2 are needed"):
            call([1])
        for enough in ([1, 1], [1, 1, 1], [[1], [1]]):                 # the null context is what is refused here
            with pytest.raises(pc.PackCacheError):
                call(enough)
    with pytest.raises(ValueError):
        pc._native().plan_budget(pc.PC_LINEAR, 0.0, 1, 0, 0, np.array([5, 5], np.int32), np.zeros(1, np.int32))


def test_current_stream_without_torchs_private_call(monkeypatch):
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: type("S", (), {"cuda_stream": 7}))
    assert pc._stream(None) == 7 and pc._stream(5) == 5


def test_native_module_is_the_one_of_this_interpreter():
    """Another interpreter's build is not importable here, nor this one there."""
    assert build.PYLIB.endswith(importlib.machinery.EXTENSION_SUFFIXES[0]) and pc._native().__file__ == build.PYLIB
