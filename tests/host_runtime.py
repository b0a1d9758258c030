"""The library's host code over a CUDA runtime that runs nothing (host_runtime.cpp): what is refused, in which order work is
enqueued, on which device and stream, and what is left behind when a call of the runtime fails, on a machine without a GPU."""
from __future__ import annotations

import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2601_04359_b200 import binding as pc
from paper_2601_04359_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))
CALLBACK = C.CFUNCTYPE(None)
DEVICE, PINNED = 2, 1                                     # cudaMemoryType


class Runtime:
    def __init__(self, path):
        self.lib = C.CDLL(path)
        self.open = []                                    # contexts and windows, closed while the binding still uses this library
        self.lib.rt_log.restype = C.c_char_p
        self.lib.rt_memory.argtypes = [C.c_void_p, C.c_size_t, C.c_int, C.c_int]
        self.lib.rt_fail.argtypes = [C.c_char_p, C.c_int]

    def log(self):
        return self.lib.rt_log().decode().splitlines()

    def reset(self):
        self.lib.rt_reset()

    def fail(self, name, after=0):
        self.lib.rt_fail(name.encode(), after)

    def device(self, d):
        self.lib.cudaSetDevice(d)

    def memory(self, *tensors, kind=DEVICE, device=0):
        for t in tensors:
            self.lib.rt_memory(t.data_ptr(), t.numel() * t.element_size(), kind, device)


@pytest.fixture(scope="session")
def _library(tmp_path_factory):
    """The library's sources, host code only in earnest (device code stops at PTX), linked with the runtime above."""
    at = tmp_path_factory.mktemp("host_runtime")
    jobs, objs = [], []
    for f in build.SOURCES:
        objs.append(str(at / (f + ".o")))
        jobs.append(subprocess.Popen([build._nvcc(), "-gencode", "arch=compute_100a,code=compute_100a", "-O1", "-std=c++17", "-Xcompiler",
                                      "-fPIC", "-I", build.INCLUDE, "-c", "-o", objs[-1], os.path.join(build.CSRC, f)]))
    assert [j.wait() for j in jobs] == [0] * len(jobs)
    cuda = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    path = str(at / "libhost.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", cuda, "-Wl,-Bsymbolic", "-o", path,
                           os.path.join(HERE, "host_runtime.cpp")] + objs)
    return path


@pytest.fixture()
def rt(_library, monkeypatch):
    """The runtime, with the binding's ctypes calls going to the library over it."""
    monkeypatch.setattr(build, "LIB", _library)
    monkeypatch.setattr(pc, "_lib", None)
    r = Runtime(_library)
    r.reset()
    r.device(0)
    yield r
    for x in reversed(r.open):
        x.close()
    r.reset()
    r.device(0)


class Case:
    """A context, a window over two history buffers and one frame, all in host memory that stands in for the device's."""

    def __init__(self, rt, *, heads=(24, 8, 128), n=130, total=200, window=4, anchors=37, max_keys=0, max_q=0):
        hq, hk, d = heads
        self.rt, self.n, self.heads = rt, n, heads
        bf = torch.bfloat16
        seg = lambda cap, k: pc.Segment(torch.zeros(cap, hk, d, dtype=bf), torch.zeros(cap, hk, d, dtype=bf), torch.zeros(cap, 4, dtype=torch.int32), k)
        self.ctx = pc.Context(hq, hk, d, pc.PC_BF16, 10000.0, (64, 64, 64), max_q or n, max_keys or anchors + total + 4 * n)
        self.anchors, self.bufs, self.frame = seg(anchors, anchors), [seg(total + 2 * n, 0) for _ in range(2)], seg(n, n)
        for s in [self.anchors, self.frame] + self.bufs:
            rt.memory(s.k, s.v, s.pos)
        self.window = (window, pc.PC_LINEAR, 0.0, total, 0)
        rt.open.append(self.ctx)
        self.q, self.q_pos = torch.zeros(n, hq, d, dtype=bf), torch.zeros(n, 4, dtype=torch.int32)
        self.out = torch.zeros_like(self.q)
        self.ws = {"q": torch.zeros_like(self.q), "q_pos": torch.zeros_like(self.q_pos), "out": torch.zeros_like(self.q)}

    def pin(self):
        """What a step takes from host memory and brings back there is pinned."""
        self.rt.memory(self.frame.k, self.frame.v, self.frame.pos, self.q, self.q_pos, self.out, kind=PINNED)
        return self

    def make(self):
        win = pc.Window(self.ctx, *self.window, self.anchors, self.bufs[0], self.bufs[1])
        self.rt.open.append(win)
        return win

    def step_host(self, win, **kw):
        f = {"k": self.frame.k, "v": self.frame.v, "pos": self.frame.pos}
        return win.step_host(f, self.q, self.q_pos, self.out, dict(self.ws, **kw), stream=0)


def counts(win):
    return win.state()[0].tolist()
