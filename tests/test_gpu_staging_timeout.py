"""A poll limit of one: the wait for a staged chunk or for the chunks before it
may give up at once.  The compressor then reports LZ_ERR_TIMEOUT (or LZ_OK when
no wait gave up) and finishes, also inside long matches, whose lengths are
measured after the wait; the context compresses exactly afterwards."""
from __future__ import annotations

import time

import numpy as np
import pytest
import torch

import oracle
from paper_2304_07342_gb300 import lz, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wpb", [0, 1])
@pytest.mark.parametrize("kind", ["zeros", "runs", "codes"])
def test_poll_limit_of_one(kind, wpb):
    r = np.random.default_rng(5)
    n = 200 * 2048
    x = {"zeros": np.zeros(n, np.uint16),
         "runs": np.repeat(r.integers(0, 9, n // 100 + 1), 100)[:n].astype(np.uint16),
         "codes": synth.quant_codes_laplace(n, seed=4)}[kind]
    P = lz.Params(2, 4096, 128, 3, 255)
    ref = oracle.compress(x, oracle.Params(2, 4096, 128, 3, 255))
    codec = G.codec()
    try:
        d = G.to_dev(x)
        out = torch.empty(lz.lz_compressed_bound(d.numel(), P), dtype=torch.uint8, device="cuda")
        nb = torch.zeros(1, dtype=torch.int64, device="cuda")
        st = torch.cuda.current_stream().cuda_stream

        def run():
            lz.lz_compress_ex(codec.ctx, d.data_ptr(), d.numel(), P, out.data_ptr(), out.numel(),
                              nb.data_ptr(), st, warps_per_block=wpb)
            return codec.sync()

        lz.lz_set_test_hooks(codec.ctx, spin_limit=1)
        for _ in range(20):
            t = time.perf_counter()
            status = run()
            assert status in (lz.LZ_OK, lz.LZ_ERR_TIMEOUT)
            assert time.perf_counter() - t < 5.0
            if status == lz.LZ_OK:
                assert np.array_equal(out[:int(nb.item())].cpu().numpy(), ref)
        lz.lz_set_test_hooks(codec.ctx)
        assert run() == lz.LZ_OK
        assert np.array_equal(out[:int(nb.item())].cpu().numpy(), ref)
    finally:
        codec.close()
