"""The parse by equality masks against the oracle where it can go wrong:
matches that end around the rows it keeps (two slabs of 32 positions) or run
on far past them, every number of varying symbol bits, windows that are not
whole words, chunk lengths around a slab, the parameters at the edge of its
route, and stored chunks whose input the record was written over.  Every case
runs with one warp per chunk (a stated launch shape) and with a block per
chunk (what few chunks take).  Streams are compared byte for byte."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_2304_07342_gb300 import lz
from tests import gpu_util as G
from tests import test_gpu_literal_precheck as precheck

pytestmark = pytest.mark.gpu

DT = {1: np.uint8, 2: np.uint16, 4: np.uint32}


@pytest.fixture(scope="module")
def codec():
    c = G.codec()
    yield c
    c.close()


def _compress(codec, d, P, wpb, match=lz.LZ_MATCH_EXACT, version=1):
    out = torch.empty(lz.lz_compressed_bound(d.numel(), P), dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    lz.lz_compress_ex(codec.ctx, d.data_ptr(), d.numel(), P, out.data_ptr(), out.numel(),
                      nb.data_ptr(), torch.cuda.current_stream().cuda_stream, match=match,
                      version=version, warps_per_block=wpb)
    assert codec.sync() == lz.LZ_OK
    return out[:int(nb.item())].cpu().numpy()


def _check(codec, x, S, C, W, m, M=255, version=1, overlap=False, offset=0):
    match = lz.LZ_MATCH_OVERLAP if overlap else lz.LZ_MATCH_EXACT
    mode = oracle.MATCH_OVERLAP if overlap else oracle.MATCH_EXACT
    ref = oracle.compress(x, oracle.Params(S, C, W, m, M), mode=mode, version=version)
    d = G.to_dev(x, offset)
    for wpb in (0, 1):
        got = _compress(codec, d, lz.Params(S, C, W, m, M), wpb, match, version)
        assert np.array_equal(got, ref), (wpb, G.first_difference(got, ref))
    assert np.array_equal(G.gpu_decompress(codec, ref), np.asarray(x).view(np.uint8).reshape(-1))


def _random(n, S, seed, bits=None):
    r = np.random.default_rng(seed)
    return r.integers(0, 1 << (bits or 8 * S), n, dtype=np.uint64).astype(DT[S])


@pytest.mark.parametrize("S,W", [(1, 128), (1, 300), (2, 128), (2, 256), (2, 512), (4, 97), (4, 256)])
@pytest.mark.parametrize("length", [31, 32, 33, 63, 64, 65, 96, 97, 128, 255])
def test_planted_matches(codec, S, W, length):
    """One repeat of `length` symbols per start inside a slab, at the largest
    offset that holds it."""
    n = min(length, W)
    C = 8192
    x = _random(40 * (C // S), S, seed=S * 1000 + length)
    for i in range(40):
        at = i * (C // S) + W + 40 + i  # every place in a slab
        x[at:at + n] = x[at - W:at - W + n]
    _check(codec, x, S, C, W, 3)


@pytest.mark.parametrize("S", [1, 2, 4])
@pytest.mark.parametrize("bits", [1, 2, 4, 5, 6, 7, 8, 9, 16, 17, 32])
def test_varying_bits(codec, S, bits):
    if bits > 8 * S:
        pytest.skip("more bits than the symbol has")
    x = _random(9000, S, seed=bits, bits=min(bits, 10)).astype(np.uint64)
    r = np.random.default_rng(bits)
    wide = r.integers(0, 1 << bits, 64, dtype=np.uint64)  # a few values over all the bits
    x = wide[x % 64].astype(DT[S]) if bits > 6 else x.astype(DT[S])
    _check(codec, x, S, 2048, 128, 3)


@pytest.mark.parametrize("S,W,m", [(1, 31, 3), (1, 1, 2), (2, 33, 2), (2, 64, 32), (2, 65, 33),
                                   (1, 256, 2), (1, 257, 2), (1, 511, 3), (1, 513, 3),
                                   (2, 512, 2), (4, 512, 1), (2, 128, 1), (4, 300, 2)])
@pytest.mark.parametrize("C", [16, 112, 2032, 4096])
def test_edges_of_the_route(codec, S, W, m, C):
    r = np.random.default_rng(W + m + C)
    x = np.repeat(r.integers(0, 5, 6000), r.integers(1, 4, 6000))[:6001].astype(DT[S])
    x[2000:3500] = np.tile(x[1900:1950], 30)  # long matches
    _check(codec, x, S, C, W, m)
    _check(codec, x, S, C, W, m, M=max(m, 40))
    _check(codec, x, S, C, W, m, version=2, overlap=True)


@pytest.mark.parametrize("S", [1, 2, 4])
def test_stored_chunks_with_pointers(codec, S):
    """Version 2: chunks with one short pointer, whose record is no smaller
    than the chunk, keep their input; the input ends in a tail and starts at
    an odd address."""
    x = _random(5 * 4096 // S + 100, S, seed=S)
    for c in range(5):
        at = c * (4096 // S) + 300
        x[at:at + 3] = x[at - 100:at - 97]
    raw = np.concatenate([x.view(np.uint8), np.arange(S - 1, dtype=np.uint8)])
    for offset in (0, 1):
        _check(codec, raw, S, 4096, 128, 3, version=2, offset=offset)


@pytest.mark.parametrize("case", precheck.CASES[::3])
def test_literal_precheck_one_warp_per_chunk(codec, case):
    """The pre-check's planted repeats with the launch that has one."""
    S, C, W, m, target, d, length = case
    x = precheck.distinct_random(2 * (C // S) + 11, S, seed=target + d)
    at = C // S + target
    n = max(0, min(length, 2 * (C // S) - at))
    for i in range(n):
        if target - d + i >= 0:
            x[at + i] = x[at - d + i]
    _check(codec, x, S, C, W, m)


@pytest.mark.parametrize("S,C,W,m", [(1, 4096, 128, 3), (2, 4096, 128, 3), (4, 4096, 256, 2)])
def test_either_side_of_the_line(codec, S, C, W, m):
    """Sizes around the line between a block and a warp per chunk: the
    streams of the two launches are the same bytes."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for chunks in (sms * 10, sms * 14, sms * 20):
        r = np.random.default_rng(chunks)
        v = r.integers(0, 40, chunks * C // S + 5)
        x = np.repeat(v, r.integers(1, 4, v.size))[:v.size].astype(DT[S])
        d = G.to_dev(x)
        P = lz.Params(S, C, W, m)
        a, b = _compress(codec, d, P, 0), _compress(codec, d, P, 1)
        assert np.array_equal(a, b)


def test_batch_with_many_chunks(codec):
    """A batch whose classes fill the GPU with one warp per chunk, and one
    small class beside them: every item equals its own call."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    params = [lz.Params(1, 2048, 64, 3), lz.Params(2, 2048, 128, 3), lz.Params(4, 2048, 256, 2),
              lz.Params(1, 2048, 512, 3), lz.Params(2, 2048, 1024, 3), lz.Params(2, 2048, 128, 3)]
    r = np.random.default_rng(0)
    ins, outs, desc = [], [], []
    nbs = torch.zeros(len(params), dtype=torch.int64, device="cuda")
    for i, P in enumerate(params):
        n = (sms * 20 if i != 3 else 40) * 2048 // P.S + 3
        v = r.integers(0, 40, n)
        x = np.repeat(v, r.integers(1, 4, n))[:n].astype(DT[P.S])
        ins.append(G.to_dev(x))
        outs.append(torch.zeros(lz.lz_compressed_bound(x.nbytes, P), dtype=torch.uint8, device="cuda"))
        desc.append((ins[i].data_ptr(), x.nbytes, outs[i].data_ptr(), outs[i].numel(),
                     nbs.data_ptr() + 8 * i, P))
    st = torch.cuda.current_stream().cuda_stream
    b = lz.lz_batch_create(codec.ctx, desc, stream=st)
    try:
        for _ in range(2):
            lz.lz_batch_run(codec.ctx, b, st)
        assert codec.sync() == lz.LZ_OK
        for d, o, n, P in zip(ins, outs, nbs.tolist(), params):
            assert np.array_equal(o[:n].cpu().numpy(), _compress(codec, d, P, 1))
    finally:
        lz.lz_batch_destroy(b, st)
