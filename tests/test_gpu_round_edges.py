"""The decoder's rounds of 128 tokens and positions and the Huffman stage's
rings and look-back, at the sizes around their edges, against the oracle."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_2304_07342_gb300 import lz, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

DT = {1: np.uint8, 2: np.uint16, 4: np.uint32}


@pytest.fixture(scope="module")
def codec():
    c = G.codec()
    yield c
    c.close()


@pytest.mark.parametrize("S,C,W", [(1, 4096, 128), (1, 4096, 300), (2, 4096, 256), (2, 4096, 300),
                                   (4, 8192, 256), (4, 32768, 512), (1, 32768, 1024)])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 127, 128, 129, 131, 255, 257, 1500])
def test_decoder_rounds(codec, S, C, W, n):
    """Chunks of n symbols: literals, short and long pointers, and in overlap
    mode chains of every depth inside a round."""
    r = np.random.default_rng(n)
    kinds = {
        "codes": np.repeat(r.integers(0, 6, n), r.integers(1, 4, n))[:n],
        "const": np.full(n, 9),
        "period": np.arange(n) % 5,
        "wide": r.integers(0, 200, n),
    }
    for name, v in kinds.items():
        x = v.astype(DT[S])
        P = oracle.Params(S, C, W, 3 if S < 4 else 2, 255)
        for version, mode in ((1, oracle.MATCH_EXACT), (2, oracle.MATCH_OVERLAP)):
            s = oracle.compress(x, P, mode=mode, version=version)
            for offset in (0, 1):
                assert np.array_equal(G.gpu_decompress(codec, s, out_offset=offset),
                                      x.view(np.uint8)), (name, version, offset)


def _huff(codec, x, in_offset=0, out_offset=0):
    d = G.to_dev(x, in_offset)
    st = torch.cuda.current_stream().cuda_stream
    cap = lz.lz_huff_bound(x.size)
    out = torch.full((cap,), 0x5A, dtype=torch.uint8, device="cuda")
    nb = torch.zeros(1, dtype=torch.int64, device="cuda")
    lz.lz_huff_compress(codec.ctx, d.data_ptr() if x.size else 0, x.size, out.data_ptr(), cap,
                        nb.data_ptr(), st)
    assert codec.sync() == lz.LZ_OK
    got = out[:int(nb.item())].cpu().numpy()
    ref = oracle.huff_compress(x)
    assert np.array_equal(got, ref)
    back = torch.zeros(x.size + out_offset + 16, dtype=torch.uint8, device="cuda")
    lz.lz_huff_decompress(codec.ctx, out.data_ptr(), got.size, back.data_ptr() + out_offset,
                          max(1, x.size), nb.data_ptr(), st)
    assert codec.sync() == lz.LZ_OK
    assert np.array_equal(back[out_offset:out_offset + x.size].cpu().numpy(), x)
    assert not back[out_offset + x.size:].any() and not back[:out_offset].any()


@pytest.mark.parametrize("n", [1, 3, 23, 24, 25, 31, 32, 33, 55, 1023, 1024, 1025, 4095, 4096, 4097,
                               8191, 32768, 32769, 33 * 32768 + 1, 70 * 32768 - 1023])
@pytest.mark.parametrize("kind", ["codes", "skewed", "bytes", "two", "one"])
def test_huffman_edges(codec, n, kind):
    """Ends of sub-blocks, warps' strings and blocks, a look-back over more
    than one window; codes of 1 to 12 bits (one to three symbols a lookup)."""
    r = np.random.default_rng(n)
    if kind == "codes":
        x = synth.quant_codes_laplace(n // 2 + 1, seed=3).view(np.uint8)[:n]
    elif kind == "skewed":  # counts about doubling: the length limit binds
        x = np.minimum(r.geometric(0.5, n), 40).astype(np.uint8)
    elif kind == "bytes":
        x = r.integers(0, 256, n).astype(np.uint8)
    elif kind == "two":
        x = (r.random(n) < 0.3).astype(np.uint8) * 200
    else:
        x = np.full(n, 77, np.uint8)
    _huff(codec, x)
    if n <= 33 * 32768:
        _huff(codec, x, in_offset=5, out_offset=3)
