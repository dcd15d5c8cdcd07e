"""The autotuner's trials run the launch that large buffers take: the library's
own choice is timed with one warp per chunk like the stated shapes, also on a
sample that would take a block per chunk by itself."""
from __future__ import annotations

import pytest
import torch

from paper_2304_07342_gb300 import lz, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def test_trials_compare_like_with_like():
    codec = G.codec()
    try:
        x = synth.quant_codes_laplace(1 << 19, seed=5)  # 1 MiB: a block per chunk by size
        d = G.to_dev(x)
        ratios = []
        for _ in range(5):
            P, wpb, trials = lz.lz_autotune_ex(codec.ctx, d.data_ptr(), d.numel(), 2)
            shapes = trials[16:]
            assert shapes[0]["warps_per_block"] == 0 and len(shapes) > 1
            ratios.append(shapes[0]["ms"] / min(t["ms"] for t in shapes[1:]))
        # (a block per chunk takes about a third of the time here)
        assert sorted(ratios)[2] > 0.7, ratios
    finally:
        codec.close()
