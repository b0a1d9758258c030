"""Timed cases of the PackCache path: one video frame of one layer (or of a stack of layers) through the calls that a
generation loop makes, from the 64-token fp32 frame of the smallest configuration to a 28-layer frame over 47 history
frames, with every way of using the cache: one-shot compaction every frame, attention over the whole cache, several passes
over one prepared cache, retention guided by attention mass, a cache mask, and the cache window on the device and from
host memory.

A case is a dict of plain values.  ``path`` names the way of using the library; the rest are sizes: query / KV heads and
head dimension, storage type, text tokens, the token grid of a frame, history frames, tokens to retain (``total``), newest
frames kept whole, and the decay kernel.  Inputs are what a model's layer would bring: unit-variance Q, K and V, for bf16
with a +-4 bias on 2 % of the K and V channels, and (t, h, w) coordinates scaled by (4, 8, 8)."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2601_04359_b200 import binding as pc

DECAY = {"geometric": pc.PC_GEOMETRIC, "closed_half": pc.PC_CLOSED_HALF, "linear": pc.PC_LINEAR, "halflife": pc.PC_HALFLIFE}
T_STEP = 4                                             # temporal coordinate units per frame


def _case(name, path, frames, total, *, heads=(24, 8, 128), dtype="bf16", n_text=128, grid=(24, 42), keep_full=0,
          decay=("halflife", 4.0), layers=1, passes=1):
    c = {"path": path, "q_heads": heads[0], "kv_heads": heads[1], "head_dim": heads[2], "dtype": dtype, "n_text": n_text,
         "rows": grid[0], "cols": grid[1], "frames": frames, "total": total, "keep_full": keep_full, "decay": decay[0],
         "param": decay[1], "layers": layers, "passes": passes}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest configuration: fp32, 64-token frames, closed-form decay; a step here is latency and launches
        _case("step_tiny_f32", "step", 6, 128, heads=(4, 2, 64), dtype="f32", n_text=32, grid=(8, 8), decay=("closed_half", 0.5)),
        # a small bf16 clip with ragged tile ends (135-token frames): thumbnails, tests, the first frames of a generation
        _case("step_small_bf16", "step", 5, 300, n_text=37, grid=(9, 15), keep_full=1, decay=("halflife", 2.0)),
        # an ordinary frame early in a generation: 12 history frames, a quarter of them kept, linear decay
        _case("step_12_frames", "step", 12, 3024, decay=("linear", 0.0)),
        # a late frame of a 48-frame generation, two newest frames whole: the headline step
        _case("step_47_frames", "step", 47, 8064, keep_full=2),
        # a high-resolution frame: 4032 tokens per frame, 11 history frames, two frames' worth of tokens kept
        _case("step_high_res", "step", 11, 8417, n_text=249, grid=(48, 84), decay=("halflife", 2.0)),
        # the same late frame through a whole stack of 28 layers, each with its own cache and context
        _case("stack_28_layers", "step", 47, 11844, layers=28),
        # no compaction: the frame attends to everything generated so far and to itself (what the cache is measured against,
        # and what every frame does until the cache is full)
        _case("attend_whole_cache", "attend", 47, 0),
        # a frame that is generated over several passes over one unchanged compacted cache: keys prepared once, five passes
        _case("passes_24_frames", "passes", 24, 6048, passes=5),
        # retention guided by attention: select on the masses the last frame left, pack, attend, and this frame's masses
        _case("guided_12_frames", "guided", 12, 3024, decay=("linear", 0.0)),
        # scoring under a cache mask, then pack and attention (with the current frame) by separate calls
        _case("masked_24_frames", "masked", 24, 6048),
        # the sliding cache window in its steady state: append the finished frame, then update and attend in one call
        _case("window_24_frames", "window", 24, 8064, keep_full=2),
        # the same from pinned host buffers: frame and queries uploaded, output downloaded every step
        _case("window_host_24_frames", "window_host", 24, 8064, keep_full=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.12:
        # fp32: small frames, head_dim 64
        grid = (_log_int(rng, 3, 20), _log_int(rng, 3, 20))
        frames = _log_int(rng, 1, 12)
        n = grid[0] * grid[1]
        total = max(1, int(rng.uniform(0.1, 0.6) * frames * n))
        return _case("", "step", frames, total, heads=(4, 2, 64), dtype="f32", n_text=_log_int(rng, 4, 64), grid=grid,
                     decay=rng.choice([("closed_half", 0.5), ("geometric", 0.7)]))
    path = rng.choice(["step", "step", "step", "attend", "passes", "guided", "masked", "window", "window_host"])
    heads = rng.choice([(24, 8, 128), (24, 8, 128), (24, 8, 128), (32, 8, 128), (16, 4, 128), (8, 8, 128), (24, 12, 128), (32, 16, 128)])
    rows = _log_int(rng, 4, 48)
    grid = (rows, max(4, min(84, int(rows * rng.uniform(1.0, 2.0)))))
    n = grid[0] * grid[1]
    most = max(2, min(47, 48000 // n))
    frames = max(2, min(most, _log_int(rng, 2, 48)))
    n_text = _log_int(rng, 16, 250)
    keep_full = rng.choice([0, 0, 1, 2]) if frames >= 8 else 0
    lo, hi = max(0.05, (keep_full + 0.5) / frames), 0.6
    total = max(frames, min(12096, int(rng.uniform(min(lo, hi), hi) * frames * n)))
    total = max(total, keep_full * n)
    decay = rng.choice([("linear", 0.0), ("halflife", float(rng.choice([4, 8])))])
    if path in ("window", "window_host"):
        # a decay that leaves every frame of the window a share, so that exactly one frame leaves per step
        frames = min(frames, 24, int(0.6 * n) - 1)
        total = max(frames * (frames + 1), min(total, int(0.6 * frames * n)))
        keep_full = 0
        decay = ("linear", 0.0)
    passes = rng.randint(2, 8) if path == "passes" else 1
    while True:
        c = _case("", path, frames, total, heads=heads, n_text=n_text, grid=grid, keep_full=keep_full, decay=decay, passes=passes)
        if work(c)["flops"] <= 4e12:                       # no more than the 28-layer frame
            return c
        if passes > 2:
            passes -= 1
        else:
            frames -= 1


# ---------------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------------
class _Inputs:
    """Seeded tensors of one layer on the GPU."""

    def __init__(self, c, seed, layer=0):
        self.c = c
        self.dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
        self.gen = torch.Generator(device="cuda").manual_seed((int(seed) * 1000 + layer) % (1 << 62))
        slots = c["kv_heads"] * c["head_dim"]
        self.bias = [self._bias(slots) if c["dtype"] == "bf16" else None for _ in range(2)]
        self.n = c["rows"] * c["cols"]

    def _bias(self, slots):
        b = torch.zeros(slots, device="cuda")
        pick = torch.randperm(slots, generator=self.gen, device="cuda")[:max(1, round(0.02 * slots))]
        b[pick] = 4.0 * (2.0 * torch.randint(0, 2, pick.shape, generator=self.gen, device="cuda") - 1.0)
        return b.view(self.c["kv_heads"], self.c["head_dim"])

    def _gauss(self, n, heads, bias=None):
        x = torch.randn((n, heads, self.c["head_dim"]), generator=self.gen, device="cuda")
        return (x if bias is None else x.add_(bias)).to(self.dt)

    def queries(self):
        return self._gauss(self.n, self.c["q_heads"])

    def kv(self, n):
        return self._gauss(n, self.c["kv_heads"], self.bias[0]), self._gauss(n, self.c["kv_heads"], self.bias[1])

    def frame_pos(self, f, tag0):
        """[n][4] coordinates of the visual tokens of frame f (0 = conditioning image)."""
        c = self.c
        i = torch.arange(self.n, dtype=torch.int32, device="cuda")
        t = torch.full_like(i, c["n_text"] + T_STEP * f)
        return torch.stack([t, 8 * (i // c["cols"]), 8 * (i % c["cols"]), tag0 + i], dim=1).to(torch.int32).contiguous()

    def anchors(self):
        """Text tokens and the conditioning image."""
        n_text = self.c["n_text"]
        i = torch.arange(n_text, dtype=torch.int32, device="cuda")
        pos = torch.cat([torch.stack([i, i, i, i], dim=1), self.frame_pos(0, n_text)])
        k, v = self.kv(n_text + self.n)
        return pc.Segment(k, v, pos.to(torch.int32).contiguous(), n_text + self.n)

    def history(self, frames):
        tag0 = self.c["n_text"] + self.n
        pos = torch.cat([self.frame_pos(f, tag0 + (f - 1) * self.n) for f in range(1, frames + 1)])
        k, v = self.kv(frames * self.n)
        return pc.Segment(k, v, pos, frames * self.n)

    def frame(self, f):
        k, v = self.kv(self.n)
        return pc.Segment(k, v, self.frame_pos(f, self.c["n_text"] + f * self.n), self.n)

    def empty(self, capacity):
        shape = (capacity, self.c["kv_heads"], self.c["head_dim"])
        return pc.Segment(torch.zeros(shape, dtype=self.dt, device="cuda"), torch.zeros(shape, dtype=self.dt, device="cuda"),
                          torch.zeros((capacity, 4), dtype=torch.int32, device="cuda"), 0)

    def context(self, max_keys):
        c = self.c
        max_pos = (c["n_text"] + T_STEP * (c["frames"] + 3) + 1, max(c["n_text"], 8 * c["rows"]), max(c["n_text"], 8 * c["cols"]))
        return pc.Context(c["q_heads"], c["kv_heads"], c["head_dim"], pc.PC_BF16 if c["dtype"] == "bf16" else pc.PC_F32, 10000.0,
                          max_pos, self.n, max_keys)


def _plan(c, frame_count):
    return pc.pc_plan_budget(DECAY[c["decay"]], c["param"], c["total"], c["keep_full"], frame_count)


def _layer(c, seed, layer):
    """What a generation loop holds for one layer: inputs, context, and the buffers that every frame writes."""
    x = _Inputs(c, seed, layer)
    n_src = c["frames"] * x.n
    s = {"ctx": x.context(c["n_text"] + x.n + n_src + x.n), "q": x.queries(), "q_pos": x.frame_pos(c["frames"] + 1, c["n_text"] + (c["frames"] + 1) * x.n)}
    s["cache"] = pc.Cache(x.anchors(), x.history(c["frames"]), np.full(c["frames"], x.n, np.int32))
    s["out"] = torch.zeros_like(s["q"])
    if c["path"] in ("attend", "guided", "masked"):
        s["current"] = x.frame(c["frames"] + 1)
        s["lse"] = torch.zeros((x.n, c["q_heads"]), dtype=torch.float32, device="cuda")
    if c["path"] == "masked":
        s["valid"] = (torch.rand(n_src, generator=x.gen, device="cuda") < 0.8).to(torch.uint8)
    if c["path"] != "attend":
        total = min(c["total"], n_src)
        s["scores"] = torch.zeros(n_src, dtype=torch.float32, device="cuda")
        s["sel"] = torch.zeros(total, dtype=torch.int32, device="cuda")
        s["dst"] = pc.Cache(s["cache"].anchors, x.empty(total), np.zeros(c["frames"], np.int32))
    if c["path"] == "guided":
        # attention masses of the history as the last frame left them: positive, summing to less than one
        s["last_mass"] = torch.softmax(torch.randn(n_src, generator=x.gen, device="cuda"), dim=0)
        s["mass"] = torch.zeros(c["n_text"] + x.n + total + x.n, dtype=torch.float32, device="cuda")
    if c["path"] == "passes":
        # the packed cache that the frame's passes attend to, and each pass's queries
        pc.pc_frame_step(s["ctx"], s["cache"], _plan(c, s["cache"].frame_count), 0, s["dst"], s["q"], s["q_pos"], scores=s["scores"],
                         sel_idx=s["sel"], out=s["out"])
        s["qs"] = [x.queries() for _ in range(c["passes"])]
        s["outs"] = [torch.zeros_like(s["q"]) for _ in range(c["passes"])]
    return s


def _window(c, seed):
    """A cache window brought to its steady state (one frame leaves for every one that is appended)."""
    x = _Inputs(c, seed)
    ctx = x.context(c["n_text"] + x.n + c["total"] + 2 * x.n + c["frames"] * x.n)
    cap = max(c["total"], c["frames"]) + 2 * x.n
    bufs = x.empty(cap), x.empty(cap)
    win = pc.Window(ctx, c["frames"], DECAY[c["decay"]], c["param"], c["total"], c["keep_full"], x.anchors(), bufs[0], bufs[1],
                    rebase=True, t_step=T_STEP)
    s = {"ctx": ctx, "win": win, "bufs": bufs, "total": c["total"], "out": torch.zeros((x.n, c["q_heads"], c["head_dim"]), dtype=x.dt, device="cuda")}
    q = x.queries()
    for f in range(1, c["frames"] + 3):
        at = min(f, c["frames"] + 1)                       # past W frames the window slides and the newest frame stays at W + 1
        win.append(x.frame(at))
        win.step(q, x.frame_pos(at + 1 if f <= c["frames"] else at, 0), out=s["out"])
    s["frame"] = x.frame(c["frames"] + 1)
    s["q"], s["q_pos"] = x.queries(), x.frame_pos(c["frames"] + 1, 0)
    if c["path"] == "window_host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        f = s["frame"]
        s["ws"] = {"q": torch.zeros_like(s["q"]), "q_pos": torch.zeros_like(s["q_pos"]), "out": s["out"]}
        s["frame"] = {"k": pin(f.k), "v": pin(f.v), "pos": pin(f.pos)}
        s["q"], s["q_pos"] = pin(s["q"]), pin(s["q_pos"])
        s["out"] = torch.zeros(s["out"].shape, dtype=x.dt).pin_memory()
    s["active"] = win.state()[2]
    torch.cuda.synchronize()
    return s


def prepare(case, seed):
    if case["path"] in ("window", "window_host"):
        return dict(_window(case, seed), case=case)
    return {"case": case, "layers": [_layer(case, seed, i) for i in range(case["layers"])]}


# ---------------------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------------------
def _packed(dst):
    n = dst.history.n_tokens
    return {"k": dst.history.k[:n], "v": dst.history.v[:n], "pos": dst.history.pos[:n]}


def _step(c, s):
    pc.pc_frame_step(s["ctx"], s["cache"], _plan(c, s["cache"].frame_count), 0, s["dst"], s["q"], s["q_pos"], scores=s["scores"],
                     sel_idx=s["sel"], out=s["out"])
    return dict(_packed(s["dst"]), out=s["out"], scores=s["scores"], sel=s["sel"])


def _attend(c, s):
    pc.pc_attend_frame(s["ctx"], s["cache"], s["current"], s["q"], s["q_pos"], out=s["out"], lse=s["lse"])
    return {"out": s["out"], "lse": s["lse"]}


def _passes(c, s):
    pc.pc_attend_prepare(s["ctx"], s["dst"])
    for q, out in zip(s["qs"], s["outs"]):
        pc.pc_attend_prepared(s["ctx"], q, s["q_pos"], out=out)
    return s["outs"]


def _guided(c, s):
    budget = _plan(c, s["cache"].frame_count)
    pc.pc_score(s["ctx"], s["cache"], None, None, budget, scores_override=s["last_mass"], sel_idx=s["sel"])
    pc.pc_compact(s["ctx"], s["cache"], s["sel"], budget, T_STEP, s["dst"])
    pc.pc_attend_frame(s["ctx"], s["dst"], s["current"], s["q"], s["q_pos"], out=s["out"], lse=s["lse"])
    pc.pc_attend_mass(s["ctx"], s["lse"], s["mass"].shape[0], mass=s["mass"])
    return dict(_packed(s["dst"]), out=s["out"], lse=s["lse"], mass=s["mass"], sel=s["sel"])


def _masked(c, s):
    budget = _plan(c, s["cache"].frame_count)
    pc.pc_score(s["ctx"], s["cache"], s["q"], s["q_pos"], budget, valid=s["valid"], scores=s["scores"], sel_idx=s["sel"])
    pc.pc_compact(s["ctx"], s["cache"], s["sel"], budget, T_STEP, s["dst"])
    pc.pc_attend_frame(s["ctx"], s["dst"], s["current"], s["q"], s["q_pos"], out=s["out"], lse=s["lse"])
    return dict(_packed(s["dst"]), out=s["out"], lse=s["lse"], scores=s["scores"], sel=s["sel"])


PATHS = {"step": _step, "attend": _attend, "passes": _passes, "guided": _guided, "masked": _masked}


def run(state):
    c = state["case"]
    if c["path"] in ("window", "window_host"):
        win = state["win"]
        if c["path"] == "window":
            win.append(state["frame"])
            win.step(state["q"], state["q_pos"], out=state["out"])
        else:
            win.step_host(state["frame"], state["q"], state["q_pos"], state["out"], state["ws"])
        state["active"] ^= 1                               # the kept tokens moved to the other buffer
        b, n = state["bufs"][state["active"]], state["total"]
        return {"out": state["out"], "k": b.k[:n], "v": b.v[:n], "pos": b.pos[:n]}
    outs = [PATHS[c["path"]](c, s) for s in state["layers"]]
    if len(outs) == 1:
        return outs[0]
    return [o["out"] for o in outs] + [outs[-1]]           # every layer's output; the packed cache of the last


# ---------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far another correct implementation may be from it
# ---------------------------------------------------------------------------------------------------------------------
def work(case):
    c = case
    e = 2 if c["dtype"] == "bf16" else 4
    n = c["rows"] * c["cols"]
    row, q_row = c["kv_heads"] * c["head_dim"] * e, c["q_heads"] * c["head_dim"] * e
    n_anchor, n_src = c["n_text"] + n, c["frames"] * n
    total = min(c["total"], n_src)
    kept = n_anchor + total
    per_key = 4 * n * c["q_heads"] * c["head_dim"]                       # Q K^T and P V of one key
    io = n * (2 * q_row + 16)                                            # queries in, outputs out
    score = n_src * (row + 16 + 4)                                       # every history key once, its score
    pack = total * (4 * row + 2 * 16 + 4)                                # kept K and V rows read and written, index
    anchors = n_anchor * (2 * row + 16)
    if c["path"] == "step":
        # a kept key row is read for its score already
        b, f = score + pack - total * row + anchors + io, kept * per_key + 2 * n_src * c["kv_heads"] * c["head_dim"]
    elif c["path"] == "attend":
        b, f = (n_anchor + n_src + n) * (2 * row + 16) + io + n * c["q_heads"] * 4, (n_anchor + n_src + n) * per_key
    elif c["path"] == "passes":
        b, f = kept * (2 * row + 16) + c["passes"] * io, c["passes"] * kept * per_key
    elif c["path"] == "guided":
        # the masses are one more Q K^T over the keys attended
        b = n_src * 4 + pack + anchors + n * (2 * row + 16) + io + n * c["q_heads"] * 4 + (kept + n) * 4
        f = (kept + n) * per_key * 1.5
    elif c["path"] == "masked":
        b = score + n_src + pack - total * row + anchors + n * (2 * row + 16) + io + n * c["q_heads"] * 4
        f = (kept + n) * per_key + 2 * n_src * c["kv_heads"] * c["head_dim"]
    else:
        src = c["total"] + n                                             # kept tokens and the appended frame
        b = src * (row + 16 + 4) + n * (row + 16) + c["total"] * (3 * row + 16 + 4) + anchors + io
        f = (n_anchor + c["total"]) * per_key + 2 * src * c["kv_heads"] * c["head_dim"]
    return {"bytes": float(c["layers"] * b), "flops": float(c["layers"] * f)}


def tolerance(case):
    # Against a 64-bit evaluation of the same inputs: fp32 outputs 3.9e-7 (largest difference 1.8e-6 of the larger of value and
    # rms), bf16 outputs 1.9e-3 (6.2e-3), fp32 scores 1.4e-7, log-sum-exps 8.4e-5 and masses 1.2e-4 of the bf16 path; no
    # selected index differed.  Four times that, and a near-tie that falls the other way.
    if case["dtype"] == "f32":
        return {"rel": 2e-6, "max": 1e-5, "differ": 0.002}
    return {"rel": 7.5e-3, "max": 0.025, "differ": 0.002}
