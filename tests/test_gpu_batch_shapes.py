"""Batches whose warps' slices come close to all the shared memory a block may
have, beside the descriptors that the block keeps there: they run, and every
stream is the oracle's."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2304_07342_gb300 import lz
from tests import gpu_util as G
from tests.test_gpu_mask_parse import DT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wpb", [0, 1, 2, 4])
@pytest.mark.parametrize("S,C,W,m", [(4, 25008, 256, 2), (4, 25088, 512, 2), (2, 29520, 256, 3),
                                     (2, 29648, 256, 3), (1, 12176, 512, 2), (1, 13616, 1024, 3),
                                     (1, 13664, 1024, 3)])
def test_slices_near_the_limit(S, C, W, m, wpb):
    codec = G.codec()
    try:
        st = torch.cuda.current_stream().cuda_stream
        r = np.random.default_rng(C)
        P = lz.Params(S, C, W, m)
        xs = [np.repeat(r.integers(0, 40, n), 2)[:n].astype(DT[S])
              for n in (3 * C // S + 5, C // S, 7)]
        ins = [G.to_dev(x) for x in xs]
        outs = [torch.zeros(lz.lz_compressed_bound(x.nbytes, P), dtype=torch.uint8, device="cuda")
                for x in xs]
        nbs = torch.zeros(len(xs), dtype=torch.int64, device="cuda")
        items = [(d.data_ptr(), x.nbytes, o.data_ptr(), o.numel(), nbs.data_ptr() + 8 * i, P)
                 for i, (x, d, o) in enumerate(zip(xs, ins, outs))]
        h = ctypes.c_void_p()
        opt = lz.lz_options(lz.LZ_MATCH_EXACT, 1, wpb)
        rc = lz.load().lz_batch_create_ex(codec.ctx, lz._items(items), len(items), 0,
                                          ctypes.byref(opt), st, ctypes.byref(h))
        single = lz.load().lz_compress_ex(codec.ctx, ins[0].data_ptr(), xs[0].nbytes,
                                          ctypes.byref(P.c()), ctypes.byref(opt),
                                          outs[0].data_ptr(), outs[0].numel(), nbs.data_ptr(), st)
        assert rc == single  # a shape is accepted as for a single buffer
        if rc != lz.LZ_OK:
            assert wpb > 1 and rc == lz.LZ_ERR_INVALID_ARG
            return
        try:
            lz.lz_batch_run(codec.ctx, h.value, st)
            assert codec.sync() == lz.LZ_OK
            for x, o, n in zip(xs, outs, nbs.tolist()):
                assert np.array_equal(o[:n].cpu().numpy(),
                                      oracle.compress(x, oracle.Params(S, C, W, m, 255)))
        finally:
            lz.lz_batch_destroy(h.value, st)
    finally:
        codec.close()
