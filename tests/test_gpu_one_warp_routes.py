"""The kernels with one warp per chunk on inputs small enough for a block per
chunk, by a stated launch shape: the bounds-checked build over masks and chains,
the look-back that runs out, and batches with every option -- stored chunks with
pointers, overlapping matches, tails, odd addresses -- against the oracle."""
from __future__ import annotations

import ctypes
import os
import subprocess
import sys
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2304_07342_gb300 import lz, synth
from tests import gpu_util as G
from tests.test_gpu_mask_parse import DT, _compress, _random

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHECKED = r'''
import sys
sys.path.insert(0, ROOT)
import numpy as np
import torch
import oracle
from paper_2304_07342_gb300 import build, lz, synth
lz.load(build.build(checked=True))
codec = lz.Codec(0)
st = torch.cuda.current_stream().cuda_stream
rng = np.random.default_rng(0)
def rare(n):
    x = rng.integers(0, 1 << 32, n, dtype=np.uint64)
    for i in range(5):
        x[100 + i::600] = x[70 + i::600][:x[100 + i::600].size]
    return x
kinds = {
    "quant": lambda n: synth.quant_codes_laplace(n, seed=1),
    "markov": lambda n: synth.markov_codes(n, seed=2),
    "const": lambda n: np.full(n, 7, np.uint32),
    "period": lambda n: (np.arange(n) % 5).astype(np.uint32),
    "runs": lambda n: np.repeat(rng.integers(0, 99, n // 150 + 1), 150)[:n],
    "rare": rare,
    "random": lambda n: rng.integers(0, 1 << 32, n, dtype=np.uint64),
}
grid = [(1, 2048, 128, 3), (1, 4096, 300, 2), (1, 8192, 512, 3), (2, 4096, 128, 3),
        (2, 2048, 512, 2), (2, 4096, 256, 3), (4, 8192, 256, 2), (4, 1024, 64, 1), (4, 4096, 512, 2)]
done = 0
for S, C, W, m in grid:
    dt = {1: np.uint8, 2: np.uint16, 4: np.uint32}[S]
    for name, gen in kinds.items():
        x = (np.asarray(gen(40_000 // S + 7)).astype(np.uint64) % (1 << (8 * S))).astype(dt)
        d = torch.from_numpy(x.view(np.uint8)).cuda()
        P = lz.Params(S, C, W, m)
        out = torch.empty(lz.lz_compressed_bound(d.numel(), P), dtype=torch.uint8, device="cuda")
        nb = torch.zeros(1, dtype=torch.int64, device="cuda")
        for wpb in (0, 1, 2):
            for version, match, mode in ((1, lz.LZ_MATCH_EXACT, oracle.MATCH_EXACT),
                                         (2, lz.LZ_MATCH_EXACT, oracle.MATCH_EXACT),
                                         (2, lz.LZ_MATCH_OVERLAP, oracle.MATCH_OVERLAP)):
                lz.lz_compress_ex(codec.ctx, d.data_ptr(), d.numel(), P, out.data_ptr(),
                                  out.numel(), nb.data_ptr(), st, match=match, version=version,
                                  warps_per_block=wpb)
                assert codec.sync() == lz.LZ_OK, (S, C, W, m, name, wpb, version, match)
                ref = oracle.compress(x, oracle.Params(S, C, W, m, 255), mode=mode, version=version)
                got = out[:int(nb.item())].cpu().numpy()
                assert np.array_equal(got, ref), (S, C, W, m, name, wpb, version, match)
        done += 1
print("checked", done)
'''


def test_checked_build():
    out = subprocess.run([sys.executable, "-c", CHECKED.replace("ROOT", repr(ROOT))],
                         capture_output=True, text=True, timeout=500, cwd=ROOT)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-4000:]
    assert "checked 63" in out.stdout


@pytest.mark.parametrize("kind", ["codes", "rare"])
@pytest.mark.parametrize("first_chunk", [1, 5])
def test_lookback_runs_out(kind, first_chunk):
    P = lz.Params(2, 4096, 128, 3)
    n = 64 * 2048
    if kind == "codes":
        x = synth.quant_codes_laplace(n, seed=21)
    else:
        x = _random(n, 2, 1)
        x[100::500] = x[90::500][:x[100::500].size]
    codec = G.codec()
    try:
        d = G.to_dev(x)
        out = torch.empty(lz.lz_compressed_bound(d.numel(), P), dtype=torch.uint8, device="cuda")
        nb = torch.zeros(1, dtype=torch.int64, device="cuda")
        lz.lz_set_test_hooks(codec.ctx, spin_limit=2000, first_chunk=first_chunk)
        t = time.perf_counter()
        lz.lz_compress_ex(codec.ctx, d.data_ptr(), d.numel(), P, out.data_ptr(), out.numel(),
                          nb.data_ptr(), torch.cuda.current_stream().cuda_stream, warps_per_block=1)
        assert codec.sync() == lz.LZ_ERR_TIMEOUT
        assert time.perf_counter() - t < 5.0
        lz.lz_set_test_hooks(codec.ctx)
        ref = oracle.compress(x, oracle.Params(2, 4096, 128, 3, 255))
        assert np.array_equal(_compress(codec, d, P, 1), ref)
    finally:
        codec.close()


def _dense_with_stored(S, C, seed):
    """Codes, and every fourth chunk wide values with one short pointer, whose
    record is no smaller than the chunk; a ragged end."""
    k = C // S
    r = np.random.default_rng(seed)
    x = np.repeat(np.rint(r.laplace(100, 2.0, 13 * k)), r.integers(1, 3, 13 * k))[:13 * k]
    x = x.astype(DT[S])
    wide = _random(k, S, seed)
    wide[300 % k:300 % k + 4] = wide[200 % k:200 % k + 4]
    for c in range(1, 13, 4):
        x[c * k:(c + 1) * k] = wide
    return np.concatenate([x.view(np.uint8), x.view(np.uint8)[:S * 37],
                           np.arange(S - 1, dtype=np.uint8)])


@pytest.mark.parametrize("wpb", [1, 2])
@pytest.mark.parametrize("match,version", [(lz.LZ_MATCH_EXACT, 2), (lz.LZ_MATCH_OVERLAP, 2),
                                           (lz.LZ_MATCH_EXACT, 1), (lz.LZ_MATCH_PAPER, 2)])
def test_batch_options(match, version, wpb):
    codec = G.codec()
    try:
        mode = {lz.LZ_MATCH_EXACT: oracle.MATCH_EXACT, lz.LZ_MATCH_OVERLAP: oracle.MATCH_OVERLAP,
                lz.LZ_MATCH_PAPER: oracle.MATCH_PAPER}[match]
        params = [lz.Params(1, 4096, 128, 3), lz.Params(2, 4096, 128, 3), lz.Params(4, 4096, 256, 2),
                  lz.Params(1, 4096, 512, 3), lz.Params(2, 2048, 512, 3), lz.Params(4, 8192, 512, 2),
                  lz.Params(2, 4096, 1024, 3)]
        st = torch.cuda.current_stream().cuda_stream
        ins, outs, refs, items = [], [], [], []
        nbs = torch.zeros(2 * len(params), dtype=torch.int64, device="cuda")
        for P in params:
            raw = _dense_with_stored(P.S, P.C, P.W)
            if version == 1:
                raw = raw[:raw.size - raw.size % P.S]
            for offset in (0, 1):
                ins.append(G.to_dev(raw, offset))
                outs.append(torch.zeros(lz.lz_compressed_bound(raw.size, P), dtype=torch.uint8,
                                        device="cuda"))
                refs.append(oracle.compress(raw, oracle.Params(P.S, P.C, P.W, P.m, 255), mode=mode,
                                            version=version))
                items.append((ins[-1].data_ptr(), raw.size, outs[-1].data_ptr(), outs[-1].numel(),
                              nbs.data_ptr() + 8 * len(items), P))
        h = ctypes.c_void_p()
        opt = lz.lz_options(match, version, wpb)
        assert lz.load().lz_batch_create_ex(codec.ctx, lz._items(items), len(items), 0,
                                            ctypes.byref(opt), st, ctypes.byref(h)) == lz.LZ_OK
        try:
            for _ in range(2):
                lz.lz_batch_run(codec.ctx, h.value, st)
            assert codec.sync() == lz.LZ_OK
            for ref, o, n in zip(refs, outs, nbs.tolist()):
                got = o[:n].cpu().numpy()
                assert np.array_equal(got, ref), G.first_difference(got, ref)
        finally:
            lz.lz_batch_destroy(h.value, st)
    finally:
        codec.close()
