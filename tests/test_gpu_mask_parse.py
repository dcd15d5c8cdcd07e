"""The parse by equality masks against the oracle where it can go wrong:
matches that end around the rows it keeps (two slabs of 32 positions) or run
on far past them, every number of varying symbol bits, windows that are not
whole words, chunk lengths around a slab, the parameters at the edge of its
route, and stored chunks whose input the record was written over.  Streams
are compared byte for byte."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2304_07342_gb300 import lz
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

DT = {1: np.uint8, 2: np.uint16, 4: np.uint32}


@pytest.fixture(scope="module")
def codec():
    c = G.codec()
    yield c
    c.close()


def _check(codec, x, S, C, W, m, M=255, version=1, overlap=False):
    match = lz.LZ_MATCH_OVERLAP if overlap else lz.LZ_MATCH_EXACT
    mode = oracle.MATCH_OVERLAP if overlap else oracle.MATCH_EXACT
    ref = oracle.compress(x, oracle.Params(S, C, W, m, M), mode=mode, version=version)
    d = G.to_dev(x)
    got = codec.compress_sync(d, lz.Params(S, C, W, m, M), match=match, version=version).cpu().numpy()
    assert np.array_equal(got, ref), G.first_difference(got, ref)
    assert np.array_equal(G.gpu_decompress(codec, got), np.asarray(x).view(np.uint8).reshape(-1))


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
        d = G.to_dev(raw, offset)
        P = lz.Params(S, 4096, 128, 3)
        got = codec.compress_sync(d, P, version=2).cpu().numpy()
        ref = oracle.compress(raw, oracle.Params(S, 4096, 128, 3, 255), version=2)
        assert np.array_equal(got, ref), G.first_difference(got, ref)
