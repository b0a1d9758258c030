"""Selection where its steps change: a frame of one key, around the block sizes and the cached keys, score ranges of one bin
per key and of many keys per bin, heaps of equal scores below, at and above what is settled by comparison, kept-whole
frames, and infinities that stretch the range."""
from __future__ import annotations

import numpy as np
import pytest

from .test_gpu_parity import _select_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 1023, 1025, 4032, 4097, 9000])
@pytest.mark.parametrize("kind", ["gauss", "few_ulps", "equal_heap", "outlier", "infinities"])
def test_selection_over_frame_lengths_and_score_ranges(n, kind):
    rng = np.random.default_rng(n)
    total = n + 300 + 7                                    # three frames: this one, a short one, one kept whole
    s = rng.standard_normal(total).astype(np.float32)
    if kind == "few_ulps":                                 # neighbouring floats, many keys a value
        s = (np.float32(1.0).view(np.uint32) + rng.integers(0, 40, total).astype(np.uint32)).view(np.float32)
    elif kind == "equal_heap":                             # 64 / 65 equal keys around the threshold, and everything equal
        s[:n][: min(n, 65 if n % 2 else 64)] = np.float32(0.125)
        s[n:n + 300] = np.float32(-3.0)
    elif kind == "outlier":                                # all but a few in one bin of the first histogram
        s = (1.0 + s * 1e-6).astype(np.float32)
        s[rng.integers(0, total, 3)] = np.float32(3e38)
        s[rng.integers(0, total, 3)] = np.float32(-3e38)
    elif kind == "infinities":
        s[rng.random(total) < 0.3] = -np.inf
        s[rng.random(total) < 0.1] = np.inf
    for share in (0.02, 0.5, 0.97):
        b = min(n, max(1, int(share * n)))
        _select_case([n, 300, 7], np.array([b, 123, 7]), s)
