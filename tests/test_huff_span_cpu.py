"""The Huffman decoder's check of a block's place in the stream, on the CPU:
the function the kernel calls (huf_span_ok) compiled by the host compiler, for
table entries around the stream's end and around 2^64."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#define __host__
#define __device__
#include "glz_common.h"
#include <cstdio>
int main() {
  unsigned long long s, e, b, n;
  while (std::scanf("%llu %llu %llu %llu", &s, &e, &b, &n) == 4)
    std::printf("%d\n", glz::huf_span_ok(s, e, b, n) ? 1 : 0);
}
"""


def test_block_spans(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "span.cpp", tmp_path / "span"
    src.write_text(SOURCE)
    inc = os.path.join(ROOT, "paper_2304_07342_gb300", "csrc")
    subprocess.check_call([cxx, "-std=c++17", "-I", inc, str(src), "-o", str(exe)])
    top = 1 << 64
    cases = []
    for bits_at, in_bytes in ((408, 408 + 4096), (272 + 136 * 70, 1 << 24)):
        room = in_bytes - bits_at
        ends = [0, 4, room - 4, room, room + 4, in_bytes, top - bits_at, top - bits_at + 4,
                top - bits_at + room, top - bits_at - 4, top - 4]
        for end in ends:
            for start in (0, 4, end - (1 << 20), end - 64, end - 4, end, end + 4):
                if 0 <= start < top:
                    cases.append((start, end, bits_at, in_bytes))
    out = subprocess.run([str(exe)], input="\n".join(" ".join(map(str, c)) for c in cases),
                         capture_output=True, text=True, check=True).stdout.split()
    assert len(out) == len(cases)
    for (start, end, bits_at, in_bytes), got in zip(cases, out):
        want = (start <= end and bits_at + end <= in_bytes and (end - start) % 4 == 0
                and end - start <= 1 << 20)
        assert got == str(int(want)), (start, end, bits_at, in_bytes)


def wrapping_streams():
    """A good stream of three blocks with the table entries of blocks 0 and 1
    replaced, so that block 1's [start, end) ends where bits_at + end wraps to
    a value inside the stream."""
    x = np.minimum(np.random.default_rng(3).geometric(0.1, 80_000), 255).astype(np.uint8)
    good = oracle.huff_compress(x)
    bits_at = 272 + 136 * 3
    for back in (64, 4096, 1 << 20):
        for over in (0, 4, 256):
            s = good.copy()
            end = (1 << 64) - bits_at + over
            s[272:288].view(np.uint64)[:] = [end - back, end]
            yield s


def test_oracle_rejects_wrapping_table_entries():
    n = 0
    for s in wrapping_streams():
        assert oracle.huff_decompress_status(s.tobytes())[0] == oracle.ECORRUPT
        n += 1
    assert n == 9
