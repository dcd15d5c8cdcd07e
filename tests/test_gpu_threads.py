"""Threads with a context and a stream each, whose calls use the same kernel
instance with small and large chunks: every launch succeeds and every stream is
the one a single thread gets."""
from __future__ import annotations

import threading

import numpy as np
import pytest
import torch

from paper_2304_07342_gb300 import lz, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wpb", [0, 1])
def test_chunk_sizes_side_by_side(wpb):
    x = synth.quant_codes_laplace(1 << 16, seed=3)
    base = G.codec()
    d = G.to_dev(x)
    sizes = (512, 16384, 1024, 8192)
    params = [lz.Params(2, C, 128, 3) for C in sizes]
    refs = [base.compress_sync(d, P).clone() for P in params]
    failures = []
    start = threading.Barrier(len(sizes))

    def work(P, ref):
        codec = lz.Codec(0)
        try:
            stream = torch.cuda.Stream()
            out = torch.empty(lz.lz_compressed_bound(d.numel(), P), dtype=torch.uint8, device="cuda")
            nb = torch.zeros(1, dtype=torch.int64, device="cuda")
            torch.cuda.synchronize()
            start.wait()
            for _ in range(400):
                lz.lz_compress_ex(codec.ctx, d.data_ptr(), d.numel(), P, out.data_ptr(),
                                  out.numel(), nb.data_ptr(), stream.cuda_stream,
                                  warps_per_block=wpb)
            assert lz.lz_sync(codec.ctx, stream.cuda_stream) == lz.LZ_OK
            n = int(nb.item())
            assert n == ref.numel() and torch.equal(out[:n], ref)
        except BaseException as e:  # noqa: BLE001 - reported by the main thread
            failures.append((P.C, repr(e)))
        finally:
            codec.close()

    threads = [threading.Thread(target=work, args=a) for a in zip(params, refs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    base.close()
    assert not failures, failures
