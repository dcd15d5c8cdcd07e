"""Matches that run on far past the rows the mask parse keeps, which the whole
warp follows: constant, periodic and long-run data at every window class
against the oracle, and their time against that of codes."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2304_07342_gb300 import lz
from tests import gpu_util as G
from tests.test_gpu_mask_parse import DT, _check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def codec():
    c = G.codec()
    yield c
    c.close()


@pytest.mark.parametrize("S,C,W", [(1, 4096, 32), (1, 8192, 512), (2, 4096, 64), (2, 4096, 128),
                                   (2, 4096, 200), (4, 8192, 256), (4, 8192, 480)])
def test_runs(codec, S, C, W):
    k = C // S
    r = np.random.default_rng(S + W)
    n = 3 * k + 61
    inputs = [np.zeros(n), np.arange(n) % (W - 1) % 250, np.arange(n) % 33,
              np.repeat(r.integers(0, 200, n // 90 + 1), 90)[:n],
              np.repeat(r.integers(0, 200, n // 300 + 1), 300)[:n]]
    for x in inputs:
        x = x.astype(DT[S])
        for M in (255, 254, 130, 64):
            _check(codec, x, S, C, W, 3, M=M)
        _check(codec, x, S, C, W, 3, version=2, overlap=True)


def _time(codec, d, P):
    out = torch.empty(lz.lz_compressed_bound(d.numel(), P), dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    times = []
    for _ in range(12):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        lz.lz_compress(codec.ctx, d.data_ptr(), d.numel(), P, out.data_ptr(), out.numel(),
                       nb.data_ptr(), st)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    assert codec.sync() == lz.LZ_OK
    return sorted(times[2:])[5]


@pytest.mark.parametrize("S", [2, 4])
def test_zeros_time(codec, S):
    """32 MiB of zeros at W = 512 against codes (measured: 2.0 and 2.2 times as
    long; 8 with every lane holding all words of the match)."""
    n = (32 << 20) // S
    r = np.random.default_rng(1)
    codes = np.repeat(np.rint(r.laplace(512, 2.0, n)), r.integers(1, 3, n))[:n].astype(DT[S])
    P = lz.Params(S, 8192, 512, 3)
    zeros = _time(codec, G.to_dev(np.zeros(n, DT[S])), P)
    assert zeros < 4 * _time(codec, G.to_dev(codes), P)
