"""The line between a block and a warp per chunk: where the library's own choice
used to take a block per chunk for thousands of chunks, it is not much slower
than a stated shape of one warp per chunk."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2304_07342_gb300 import lz
from tests import gpu_util as G
from tests.test_gpu_mask_parse import DT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,C,W,m,chunks", [(1, 2048, 128, 3, 3000), (2, 2048, 128, 3, 3000),
                                            (4, 2048, 256, 2, 1500), (1, 8192, 512, 3, 1000)])
def test_choice_is_no_slower(S, C, W, m, chunks):
    codec = G.codec()
    try:
        n = chunks * C // S
        r = np.random.default_rng(1)
        x = np.repeat(np.rint(r.laplace(512 if S > 1 else 128, 2.0, n)), r.integers(1, 3, n))[:n]
        d = G.to_dev(x.astype(DT[S]))
        P = lz.Params(S, C, W, m)
        out = torch.empty(lz.lz_compressed_bound(d.numel(), P), dtype=torch.uint8, device="cuda")
        nb = torch.zeros(1, dtype=torch.int64, device="cuda")
        st = torch.cuda.current_stream().cuda_stream

        def time(wpb):
            times = []
            for _ in range(12):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                lz.lz_compress_ex(codec.ctx, d.data_ptr(), d.numel(), P, out.data_ptr(),
                                  out.numel(), nb.data_ptr(), st, warps_per_block=wpb)
                b.record()
                torch.cuda.synchronize()
                times.append(a.elapsed_time(b))
            assert codec.sync() == lz.LZ_OK
            return sorted(times[2:])[5]

        # (a block per chunk took 1.2 to 1.55 times as long)
        assert time(0) < 1.15 * time(2 if C == 8192 else 4)
    finally:
        codec.close()
