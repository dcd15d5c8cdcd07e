"""The launches of a compression batch have the priority of the stream that runs
it, also those of the classes on the batch's own streams: read from the nodes of
a captured run, whose launches keep their streams' priority."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest
import torch

from paper_2304_07342_gb300 import lz
from tests import gpu_util as G
from tests.test_gpu_mask_parse import DT

pytestmark = pytest.mark.gpu

KERNEL_NODE, PRIORITY = 0, 8  # cudaGraphNodeTypeKernel, cudaLaunchAttributePriority


def _kernel_priorities(rt, graph):
    n = ctypes.c_size_t()
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    out = []
    for node in nodes:
        kind = ctypes.c_int()
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == KERNEL_NODE:
            value = (ctypes.c_int * 32)()
            assert rt.cudaGraphKernelNodeGetAttribute(ctypes.c_void_p(node), PRIORITY, value) == 0
            out.append(value[0])
    return out


def test_every_launch_has_the_streams_priority():
    lib = lz.load()
    rt = ctypes.CDLL("libcudart.so.13")
    codec = G.codec()
    try:
        params = [lz.Params(1, 4096, 128, 3), lz.Params(2, 4096, 128, 3), lz.Params(4, 8192, 256, 2)]
        r = np.random.default_rng(0)
        xs = [r.integers(0, 9, n).astype(DT[P.S]) for P in params for n in (9000, 3_000_000)]
        ps = [P for P in params for _ in range(2)]
        ins = [G.to_dev(x) for x in xs]
        outs = [torch.zeros(lz.lz_compressed_bound(x.nbytes, P), dtype=torch.uint8, device="cuda")
                for x, P in zip(xs, ps)]
        nbs = torch.zeros(len(xs), dtype=torch.int64, device="cuda")
        items = [(d.data_ptr(), x.nbytes, o.data_ptr(), o.numel(), nbs.data_ptr() + 8 * i, P)
                 for i, (x, d, o, P) in enumerate(zip(xs, ins, outs, ps))]
        high = torch.cuda.Stream(priority=-1)
        plain = torch.cuda.Stream()
        wanted = {}
        for s in (high, plain):
            prio = ctypes.c_int()
            assert rt.cudaStreamGetPriority(ctypes.c_void_p(s.cuda_stream), ctypes.byref(prio)) == 0
            wanted[s] = prio.value
        assert wanted[high] != wanted[plain]
        torch.cuda.synchronize()
        for planned in (plain, high):
            b = lz.lz_batch_create(codec.ctx, items, stream=planned.cuda_stream)
            torch.cuda.synchronize()
            try:
                for run in (high, plain, high):
                    st = ctypes.c_void_p(run.cuda_stream)
                    assert rt.cudaStreamBeginCapture(st, 0) == 0  # global mode
                    rc = lib.lz_batch_run(codec.ctx, b, run.cuda_stream)
                    graph = ctypes.c_void_p()
                    assert rt.cudaStreamEndCapture(st, ctypes.byref(graph)) == 0
                    assert rc == lz.LZ_OK
                    got = _kernel_priorities(rt, graph)
                    assert len(got) >= 3 and set(got) == {wanted[run]}, (wanted[run], got)
                    assert rt.cudaGraphDestroy(graph) == 0
                # and the runs themselves still give the streams
                lz.lz_batch_run(codec.ctx, b, high.cuda_stream)
                assert lz.lz_sync(codec.ctx, high.cuda_stream) == lz.LZ_OK
                for x, P, o, n in zip(xs, ps, outs, nbs.tolist()):
                    assert torch.equal(o[:n], codec.compress_sync(G.to_dev(x), P))
            finally:
                lz.lz_batch_destroy(b, high.cuda_stream)
                torch.cuda.synchronize()
    finally:
        codec.close()
