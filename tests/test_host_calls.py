"""Host-side behaviour of the library's calls, over a CUDA runtime that runs nothing."""
from __future__ import annotations

import ctypes as C

import numpy as np
import pytest
import torch

from paper_2601_04359_b200 import binding as pc

from .host_runtime import CALLBACK, Case, _library, counts, rt  # noqa: F401


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
