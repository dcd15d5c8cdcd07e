"""Decoding of codes of which no two fit into one lookup (bytes that all occur
about as often): against the input at the edges of rounds and sub-blocks, for
codes around that limit, for corrupt streams, and the time against codes."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_2304_07342_gb300 import lz
from tests import gpu_util as G
from tests.test_gpu_round_edges import _huff

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def codec():
    c = G.codec()
    yield c
    c.close()


@pytest.mark.parametrize("values", [256, 128, 127, 65, 64, 63, 129, 200])
@pytest.mark.parametrize("n", [300, 1023, 1024, 1025, 1031, 1032, 4097, 32768, 65536 + 1000 + 7])
def test_near_uniform(codec, values, n):
    r = np.random.default_rng(n + values)
    x = r.permutation(np.arange(n) % values).astype(np.uint8)
    _huff(codec, x)
    _huff(codec, x, in_offset=3, out_offset=5)


def test_corrupt(codec):
    x = np.random.default_rng(1).integers(0, 256, 70_000).astype(np.uint8)
    good = oracle.huff_compress(x)
    st = torch.cuda.current_stream().cuda_stream
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    out = torch.zeros(x.size, dtype=torch.uint8, device="cuda")
    bits_at = 272 + 136 * 3
    for at, flip in ((bits_at + 40, 0xFF), (272 + 24 + 4, 1), (272 + 24 + 200, 3), (good.size - 9, 0x55)):
        s = good.copy()
        s[at] ^= flip
        want = oracle.huff_decompress_status(s.tobytes())[0]
        d = G.to_dev(s)
        lz.lz_huff_decompress(codec.ctx, d.data_ptr(), d.numel(), out.data_ptr(), out.numel(),
                              nb.data_ptr(), st)
        got = codec.sync()
        assert (got == lz.LZ_ERR_CORRUPT) == (want == oracle.ECORRUPT)


def test_time(codec):
    """8 MiB of uniform bytes against codes (1.59 times as long with lookups made
    for several symbols; 1.45 is what one symbol a lookup took before them)."""
    st = torch.cuda.current_stream().cuda_stream
    n = 8 << 20
    r = np.random.default_rng(1)
    times = []
    for x in (r.integers(0, 256, n).astype(np.uint8),
              np.repeat(np.rint(r.laplace(512, 2.0, n // 2)), r.integers(1, 3, n // 2))[:n // 2]
              .astype(np.uint16).view(np.uint8)):
        d = G.to_dev(x)
        out = torch.zeros(lz.lz_huff_bound(n), dtype=torch.uint8, device="cuda")
        nb = torch.zeros(1, dtype=torch.int64, device="cuda")
        lz.lz_huff_compress(codec.ctx, d.data_ptr(), n, out.data_ptr(), out.numel(),
                            nb.data_ptr(), st)
        assert codec.sync() == lz.LZ_OK
        size, back, t = int(nb.item()), torch.zeros_like(d), []
        for _ in range(15):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            lz.lz_huff_decompress(codec.ctx, out.data_ptr(), size, back.data_ptr(), n,
                                  nb.data_ptr(), st)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        assert codec.sync() == lz.LZ_OK and torch.equal(back, d)
        times.append(sorted(t[3:])[6])
    assert times[0] < 1.5 * times[1], times
