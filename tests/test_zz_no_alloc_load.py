"""lz_compress_noalloc after its documented warm-up (one call for every symbol
size and window class): calls with another min_match, matcher route or kind of
data launch kernels whose code the warm-up has loaded, so they take no device
memory.  In a process of its own, where nothing is loaded yet."""
from __future__ import annotations

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import sys
sys.path.insert(0, ROOT)
import torch
from paper_2304_07342_gb300 import lz
n = 64 * 4096
x = torch.randint(0, 256, (n,), dtype=torch.uint8, device="cuda")
out = torch.empty(4 * n, dtype=torch.uint8, device="cuda")
nb = torch.zeros(1, dtype=torch.int64, device="cuda")
windows = (32, 64, 128, 256, 512, 1024)

def call(S, W, m):
    lz.lz_compress_noalloc(x.data_ptr(), n, lz.Params(S, 4096, W, m), out.data_ptr(), out.numel(),
                           nb.data_ptr())
    torch.cuda.synchronize()

def free():
    return torch.cuda.mem_get_info()[0]

for warm, later in ((40, 3),):
    for S in (1, 2, 4):
        for W in windows:
            call(S, W, warm)
    before = free()
    for S in (1, 2, 4):
        for W in windows:
            call(S, W, later)
    print("taken", before - free())
"""


def test_other_parameters_take_no_memory():
    out = subprocess.run([sys.executable, "-c", SCRIPT.replace("ROOT", repr(ROOT))],
                         capture_output=True, text=True, timeout=300, cwd=ROOT,
                         env={**os.environ, "CUDA_MODULE_LOADING": "LAZY"})
    assert out.returncode == 0, out.stderr[-3000:]
    assert out.stdout.split()[-2:] == ["taken", "0"], out.stdout
