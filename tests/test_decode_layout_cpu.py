"""The decoder's shared-memory slice (decode_layout, compiled by the host
compiler): as many warps on a multiprocessor as its regions allow, and regions
that hold what the phases put into them."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#define __host__
#define __device__
#include "glz_common.h"
#include <cstdio>
int main() {
  unsigned S, C, W, m;
  while (std::scanf("%u %u %u %u", &S, &C, &W, &m) == 4) {
    const unsigned offB = W <= 256 ? 1 : 2;
    const unsigned long long k = C / S;
    const glz::DecodeLayout L = glz::decode_layout(
        k, C, glz::decode_record_bound(k, S, offB, m), S == 1 && offB == 2, S * m >= 1 + offB,
        232448);
    std::printf("%u %u %u %u %u %u %u %u\n", L.per_warp, L.marks_off, L.mark_bytes, L.flags_off,
                L.flag_bytes, L.dist_off, L.hi_off, L.io_off);
  }
}
"""


def test_slices(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "layout.cpp", tmp_path / "layout"
    src.write_text(SOURCE)
    inc = os.path.join(ROOT, "paper_2304_07342_gb300", "csrc")
    subprocess.check_call([cxx, "-std=c++17", "-I", inc, str(src), "-o", str(exe)])
    cases = [(S, C, W, m) for S in (1, 2, 4) for C in (16, 112, 2048, 4096, 8192, 32768)
             for W in (64, 256, 512) for m in (1, 2, 3)]
    out = subprocess.run([str(exe)], input="\n".join(" ".join(map(str, c)) for c in cases),
                         capture_output=True, text=True, check=True).stdout.split()
    warps = {}
    for i, (S, C, W, m) in enumerate(cases):
        per_warp, marks, nmarks, flags, nflags, dist, hi, io = map(int, out[8 * i:8 * i + 8])
        k = C // S
        assert nmarks >= k and nmarks % 128 == 0 and marks + nmarks <= flags
        # flag words of up to k tokens, cleared to a round of 128; distances of a round
        assert nflags >= -(-k // 128) * 16 and flags + nflags <= hi <= io <= per_warp
        assert flags % 16 == 0 and dist % 16 == 0 and io % 16 == 0
        assert dist + 2 * 128 + 2 <= hi
        warps[S, C, W, m] = 232448 // per_warp
    # sorted 4-byte indices and 2-byte codes, as before the rounds of 128
    assert warps[4, 8192, 256, 2] >= 21
    assert warps[2, 4096, 64, 3] >= 30
