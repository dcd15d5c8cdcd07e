"""Table entries of a Huffman stream near 2^64 are reported as corrupt by the
decoder, which reads nothing for them (the check itself, on the CPU:
test_huff_span_cpu.py)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2304_07342_gb300 import lz
from tests import gpu_util as G
from tests.test_huff_span_cpu import wrapping_streams

pytestmark = pytest.mark.gpu


def test_wrapping_table_entries_are_corrupt():
    codec = G.codec()
    try:
        st = torch.cuda.current_stream().cuda_stream
        nb = torch.zeros(1, dtype=torch.int64, device="cuda")
        for s in wrapping_streams():
            d = G.to_dev(s)
            out = torch.zeros(80_000, dtype=torch.uint8, device="cuda")
            lz.lz_huff_decompress(codec.ctx, d.data_ptr(), d.numel(), out.data_ptr(), out.numel(),
                                  nb.data_ptr(), st)
            assert codec.sync() == lz.LZ_ERR_CORRUPT
    finally:
        codec.close()
