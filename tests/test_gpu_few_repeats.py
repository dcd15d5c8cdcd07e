"""Data whose symbols seldom repeat: a sample taken before the launch sends it to
the hash chains, in place of the equality masks.  Streams against the oracle
for values of all bits with few repeats, at every window class, with one warp
per chunk and a block per chunk, through a batch, and for inputs that change
between few and many repeats; and the time, which the masks take whatever the
data and the chains do not."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2304_07342_gb300 import lz
from tests import gpu_util as G
from tests.test_gpu_long_matches import _time
from tests.test_gpu_mask_parse import DT, _check, _compress, _random

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def codec():
    c = G.codec()
    yield c
    c.close()


def _planted(n, S, seed, every, length, back):
    """Wide random values; every `every` symbols a copy of `length` symbols from
    up to `back` before."""
    r = np.random.default_rng(seed)
    x = _random(n, S, seed)
    at = back + 1
    while at + length + 40 < n:
        d = int(r.integers(1, back + 1))
        for i in range(length):
            x[at + i] = x[at - d + i]
        at += int(every * (0.5 + r.random()))
    return x


def _kinds(S, n, W):
    r = np.random.default_rng(S + W)
    yield "rare", _planted(n, S, 1, 700, 5, W)
    yield "often", _planted(n, S, 2, 40, 6, min(W, 200))
    yield "edge", _planted(n, S, 3, 90, 9, W + 3)
    pool = r.integers(0, 1 << (8 * S), 300, dtype=np.uint64)
    yield "pool", pool[r.integers(0, 300, n)].astype(DT[S])
    yield "random", _random(n, S, 5)
    yield "long", _planted(n, S, 6, 900, 400, W)
    mixed = _planted(n, S, 7, 300, 8, W)
    mixed[n // 3: n // 2] = r.integers(0, 3, n // 2 - n // 3)  # many repeats half way through
    yield "mixed", mixed


@pytest.mark.parametrize("S,C,W,m", [
    (1, 4096, 128, 3), (1, 8192, 512, 3), (1, 2048, 31, 2), (1, 16384, 256, 5), (1, 4096, 257, 3),
    (2, 4096, 128, 3), (2, 4096, 64, 2), (2, 8192, 512, 2), (2, 2048, 256, 8), (2, 2032, 97, 32),
    (4, 8192, 256, 2), (4, 4096, 512, 1), (4, 4096, 33, 3), (4, 16384, 128, 2), (4, 2048, 511, 4)])
def test_against_the_oracle(codec, S, C, W, m):
    for name, x in _kinds(S, 5 * C // S + 77, W):
        _check(codec, x, S, C, W, m)
        _check(codec, x, S, C, W, m, M=max(m, 19))
        raw = np.concatenate([x.view(np.uint8), np.arange(S - 1, dtype=np.uint8)])
        _check(codec, raw, S, C, W, m, version=2, offset=1)
        _check(codec, raw, S, C, W, m, version=2, overlap=True)


@pytest.mark.parametrize("S,W", [(1, 128), (1, 512), (2, 128), (4, 256)])
@pytest.mark.parametrize("length", [1, 2, 63, 64, 127, 128, 129, 500])
def test_short_inputs(codec, S, W, length):
    for name, x in _kinds(S, 2000, min(W, 60)):
        _check(codec, x[:length].copy(), S, 4096, W, 2)


def test_mixed_data_of_many_chunks(codec):
    """Data that changes between few and many repeats every few chunks."""
    S, C, W, m = 2, 2048, 128, 3
    k = C // S
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = sms * 200
    r = np.random.default_rng(0)
    wide = _planted(n * k, S, 11, 200, 6, W).reshape(n, k)
    codes = r.integers(0, 6, (n, k)).astype(DT[S])
    dense = (np.arange(n) // 3) % 2 == 1
    x = np.where(dense[:, None], codes, wide).reshape(-1)
    ref = oracle.compress(x, oracle.Params(S, C, W, m, 255))
    for wpb in (0, 2):
        got = _compress(codec, G.to_dev(x), lz.Params(S, C, W, m), wpb)
        assert np.array_equal(got, ref), G.first_difference(got, ref)


@pytest.mark.parametrize("version,match", [(1, lz.LZ_MATCH_EXACT), (2, lz.LZ_MATCH_OVERLAP)])
@pytest.mark.parametrize("wpb", [0, 1])
def test_batch(codec, version, match, wpb):
    params = [lz.Params(1, 4096, 128, 3), lz.Params(2, 4096, 128, 3), lz.Params(4, 8192, 256, 2),
              lz.Params(1, 8192, 512, 3)]
    mode = oracle.MATCH_OVERLAP if match == lz.LZ_MATCH_OVERLAP else oracle.MATCH_EXACT
    ins, outs, desc, refs = [], [], [], []
    for P in params:
        for name, x in _kinds(P.S, 30_000 // P.S + 5, P.W):
            refs.append(oracle.compress(x, oracle.Params(P.S, P.C, P.W, P.m, 255), mode=mode,
                                        version=version))
            ins.append(G.to_dev(x))
            outs.append(torch.zeros(lz.lz_compressed_bound(x.nbytes, P), dtype=torch.uint8,
                                    device="cuda"))
            desc.append([ins[-1].data_ptr(), x.nbytes, outs[-1].data_ptr(), outs[-1].numel(), 0, P])
    nbs = torch.zeros(len(desc), dtype=torch.int64, device="cuda")
    for i, d in enumerate(desc):
        d[4] = nbs.data_ptr() + 8 * i
    st = torch.cuda.current_stream().cuda_stream
    h = ctypes.c_void_p()
    opt = lz.lz_options(match, version, wpb)
    assert lz.load().lz_batch_create_ex(codec.ctx, lz._items([tuple(d) for d in desc]), len(desc),
                                        0, ctypes.byref(opt), st, ctypes.byref(h)) == lz.LZ_OK
    b = h.value
    try:
        lz.lz_batch_run(codec.ctx, b, st)
        assert codec.sync() == lz.LZ_OK
        for ref, o, n in zip(refs, outs, nbs.tolist()):
            assert np.array_equal(o[:n].cpu().numpy(), ref)
    finally:
        lz.lz_batch_destroy(b, st)


@pytest.mark.parametrize("S,W,m", [(4, 256, 2), (2, 128, 3), (1, 128, 3)])
def test_few_repeats_take_less_time_than_many(codec, S, W, m):
    """32 MiB with a repeat every 700 symbols against codes (measured: 0.4 to
    0.6 of their time; by masks 0.8 to 1.7)."""
    r = np.random.default_rng(1)
    n = (32 << 20) // S
    codes = np.repeat(np.rint(r.laplace(512 if S > 1 else 128, 2.0, n)), r.integers(1, 3, n))[:n]
    rare = _random(n, S, 3)
    for i in range(4):
        rare[1000 + i::700] = rare[970 + i::700][:rare[1000 + i::700].size]
    P = lz.Params(S, 4096, W, m)
    few, many = (_time(codec, G.to_dev(x.astype(DT[S])), P) for x in (rare, codes))
    assert few < 0.72 * many, (few, many)
