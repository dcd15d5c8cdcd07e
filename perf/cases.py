"""Workloads of the codec's users, through its public entry points.

Inputs are drawn on the GPU from a seed, with the distributions of
``paper_2304_07342_gb300/synth.py``: uint16 quantization codes, first-order
Markov codes stored as 1-, 2- or 4-byte symbols, a smooth float32 field with
noise, sorted int32 indices, and uniform bytes.  Every output is bytes or a
byte count (streams, decoded data, sizes); there are no computed floating
numbers, so no ``exact``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2304_07342_gb300 import lz

KIB, MIB = 1 << 10, 1 << 20

# symbol size and the streams' usual size as a share of the input (for work())
SYMBOL = {"quant": 2, "markov8": 1, "markov16": 2, "markov32": 4, "field": 4, "indices": 4,
          "uniform": 1}
STREAM_SHARE = {"quant": 0.70, "markov8": 0.84, "markov16": 0.68, "markov32": 0.42, "field": 1.03,
                "indices": 1.03, "uniform": 1.13}
HUFF_SHARE = {"quant": 0.36, "markov8": 0.52, "markov16": 0.40, "markov32": 0.33, "field": 0.95,
              "indices": 0.9, "uniform": 1.0}


def listed():
    return [
        # a small array of quantization codes, as one call: latency counts
        dict(name="quant-1m-compress", op="compress", kind="quant", n=MIB, S=2, C=4096, W=128, m=3),
        dict(name="quant-1m-decompress", op="decompress", kind="quant", n=MIB, S=2, C=4096, W=128,
             m=3),
        # large nearly incompressible arrays: a float field, a sorted index column
        dict(name="field-256m-compress", op="compress", kind="field", n=256 * MIB, S=4, C=8192,
             W=256, m=2),
        dict(name="indices-512m-decompress", op="decompress", kind="indices", n=512 * MIB, S=4,
             C=8192, W=256, m=2),
        # a large array of quantization codes, both directions
        dict(name="quant-256m-compress", op="compress", kind="quant", n=256 * MIB, S=2, C=4096,
             W=128, m=3),
        dict(name="quant-256m-decompress", op="decompress", kind="quant", n=256 * MIB, S=2, C=4096,
             W=128, m=3),
        # byte codes at a higher-ratio setting; a ragged length at an odd address
        dict(name="bytes-96m-compress", op="compress", kind="markov8", n=96 * MIB + 4321, S=1,
             C=8192, W=512, m=3, offset=1),
        # 4-byte codes that compress well, written as stream version 2 with a tail
        dict(name="words-128m-compress", op="compress", kind="markov32", n=128 * MIB + 4099, S=4,
             C=4096, W=256, m=2, version=2),
        # the entropy stage on its own input, both directions
        dict(name="huff-128m-encode", op="huff_encode", kind="quant", n=128 * MIB + 5),
        dict(name="huff-128m-decode", op="huff_decode", kind="quant", n=128 * MIB + 5),
        # one admitted group of a serving loop: a compression and a
        # decompression batch over mixed requests
        dict(name="serve-64-requests", op="serve", requests=64),
        # host memory in, host memory out
        dict(name="field-128m-host", op="host", kind="field", n=128 * MIB, S=4, C=8192, W=256,
             m=2),
    ]


def _size(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    op = rng.choice(["compress", "compress", "compress", "decompress", "decompress", "huff_encode",
                     "huff_decode", "serve", "host"])
    if op == "serve":
        return dict(op=op, requests=rng.randint(4, 64))
    kind = rng.choice(["quant", "quant", "markov8", "markov16", "markov32", "field", "indices",
                       "uniform"])
    if op.startswith("huff"):
        return dict(op=op, kind=kind, n=_size(rng, 64 * KIB, 128 * MIB))
    S = rng.choice([1, 2, 4]) if kind == "uniform" else SYMBOL[kind]
    case = dict(op=op, kind=kind, S=S, C=rng.choice([2048, 4096, 4096, 8192, 16384]),
                W=rng.choice([64, 128, 256, 512]), m=2 if S == 4 else 3)
    n = _size(rng, 64 * KIB, (32 if S == 1 or case["C"] == 16384 else 128) * MIB)
    if op != "host":
        style = rng.choice(["plain", "plain", "plain", "v2", "overlap", "odd address"])
        if style in ("v2", "overlap"):
            case["version"] = 2
            case["overlap"] = style == "overlap"
        if style == "odd address":
            case["offset"] = S * rng.randint(1, 7)
    if case.get("version") != 2:
        n -= n % S
    return dict(case, n=n)


# --- inputs ---------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _laplace_codes(n, b, g):
    u = torch.rand(n, generator=g, device="cuda").sub_(0.5)
    v = torch.sign(u).mul_(torch.log1p(u.abs_().mul_(-2.0).clamp_(min=-0.9999999))).mul_(-b)
    return v.round_().add_(512).clamp_(0, 1023).to(torch.int32)


def _runs(v, keep, g):
    """v with each position repeating the value before it with probability `keep`."""
    jump = torch.rand(v.numel(), generator=g, device="cuda") >= keep
    jump[0] = True
    return v[torch.cumsum(jump, 0).sub_(1)]


def _field(n, seed, g):
    """n float32 values of a field of 512 x 256 planes (as synth.gaussian_field)."""
    nx, (ny, nz) = -(-n // (512 * 256)), (512, 256)
    full = max(512, nx)
    r = np.random.default_rng(seed)
    centre = r.uniform(0.0, 1.0, (16, 3)) * np.array([full, ny, nz], float)
    sigma, amp = r.uniform(8.0, 64.0, 16), r.normal(0.0, 1.0, 16)
    x0 = (full - nx) // 2
    axes = [torch.arange(a, b, device="cuda", dtype=torch.float32)
            for a, b in ((x0, x0 + nx), (0, ny), (0, nz))]
    acc = torch.zeros(nx, ny, nz, device="cuda")
    for c, s, a in zip(centre, sigma, amp):
        gx, gy, gz = (torch.exp((t - float(q)) ** 2 / float(-2 * s * s)) for t, q in zip(axes, c))
        acc += float(a) * gx[:, None, None] * (gy[:, None] * gz[None, :])
    acc += torch.randn(acc.shape, generator=g, device="cuda").mul_(1e-4)
    return acc.reshape(-1)[:n]


def _data(kind, n, seed):
    """n bytes of a kind, as a device uint8 tensor."""
    g = _gen(seed)
    if kind == "uniform":
        return torch.randint(0, 256, (n,), generator=g, device="cuda", dtype=torch.uint8)
    S = SYMBOL[kind]
    k = -(-n // S)
    if kind == "quant":
        v = _runs(_laplace_codes(k, 2.0, g), 0.3, g).to(torch.int16)
    elif kind == "field":
        v = _field(k, seed, g)
    elif kind == "indices":
        u = torch.rand(k, generator=g, device="cuda").clamp_(min=1e-7)
        v = torch.cumsum(torch.log(u).div_(math.log(0.7)).ceil_().clamp_(min=1).to(torch.int32), 0,
                         dtype=torch.int32)
    else:
        v = _runs(_laplace_codes(k, 4.0, g), 0.6, g)
        v = v.to(torch.uint8) if S == 1 else v.to(torch.int16) if S == 2 else v
    return v.contiguous().view(torch.uint8)[:n].clone()


def _placed(x, offset):
    """x at an address `offset` bytes past an aligned one."""
    if not offset:
        return x
    buf = torch.empty(x.numel() + offset, dtype=torch.uint8, device="cuda")
    buf[offset:].copy_(x)
    return buf[offset:]


# --- states ---------------------------------------------------------------------

_CODEC = None


def _codec():
    """The program's one codec (a context on device 0)."""
    global _CODEC
    if _CODEC is None:
        _CODEC = lz.Codec(0)
    return _CODEC


def _params(case):
    return lz.Params(case["S"], case["C"], case["W"], case["m"])


def _options(case):
    return dict(version=case.get("version", 1),
                match=lz.LZ_MATCH_OVERLAP if case.get("overlap") else lz.LZ_MATCH_EXACT)


def _zeros(n, **kw):
    return torch.zeros(max(1, n), dtype=torch.uint8, **{"device": "cuda", **kw})


def _size_word(n=1):
    return torch.zeros(n, dtype=torch.int64, device="cuda")


def prepare(case, seed):
    c = _codec()
    if case["op"] == "serve":
        return _Serve(case["requests"], seed)
    x = _placed(_data(case["kind"], case["n"], seed), case.get("offset", 0))
    s = dict(op=case["op"], codec=c, x=x, n=case["n"], nb=_size_word())
    if case["op"] == "compress":
        p = _params(case)
        return dict(s, p=p, opt=_options(case), out=_zeros(lz.lz_compressed_bound(case["n"], p)))
    if case["op"] == "decompress":
        stream = c.compress_sync(x, _params(case), **_options(case)).clone()
        return dict(s, x=stream, out=_placed(_zeros(case["n"]), case.get("offset", 0)))
    if case["op"] == "host":
        p = _params(case)
        h = torch.empty(case["n"], dtype=torch.uint8, pin_memory=True)
        h.copy_(x)
        return dict(s, x=h, p=p, out=_zeros(lz.lz_compressed_bound(case["n"], p), device="cpu",
                                            pin_memory=True))
    out = _zeros(lz.lz_huff_bound(case["n"]))
    if case["op"] == "huff_encode":
        return dict(s, out=out)
    lz.lz_huff_compress(c.ctx, x.data_ptr(), x.numel(), out.data_ptr(), out.numel(),
                        s["nb"].data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert c.sync() == lz.LZ_OK
    return dict(s, x=out[:int(s["nb"].item())].clone(), out=_zeros(case["n"]))


class _Serve:
    """A group of requests: 70 % compress, 30 % decompress, lognormal sizes, Markov
    codes of mixed symbol sizes, with the serving loop's parameters; each
    direction planned as a batch.  Sizes depend on the group size alone."""

    PARAMS = {1: lz.Params(1, 4096, 128, 3), 2: lz.Params(2, 4096, 128, 3),
              4: lz.Params(4, 8192, 256, 2)}

    def __init__(self, requests, seed):
        c, st = _codec(), torch.cuda.current_stream().cuda_stream
        sizes, sym, comp = self.mix(requests)
        self.batches, self.outs, self.keep = [], [], []
        pools = {S: _data("markov%d" % (8 * S), int(sizes.max()) + 64 * KIB, seed + S)
                 for S in (1, 2, 4)}
        r = np.random.default_rng(seed)
        for want in (True, False):
            rows, at = [], 0
            for n, S, is_comp in zip(sizes, sym, comp):
                if is_comp != want:
                    continue
                n, S, p = int(n), int(S), self.PARAMS[int(S)]
                off = 16 * int(r.integers(0, (pools[S].numel() - n) // 16 + 1))
                x = pools[S][off:off + n]
                if not want:
                    x = c.compress_sync(x, p).clone()
                cap = lz.lz_compressed_bound(n, p) if want else n
                rows.append((x, at, cap, p))
                self.keep.append(x)
                at += -(-cap // 256) * 256
            out, nb = _zeros(at), _size_word(max(1, len(rows)))
            items = [(x.data_ptr(), x.numel(), out.data_ptr() + o, cap, nb.data_ptr() + 8 * i, p)
                     for i, (x, o, cap, p) in enumerate(rows)]
            self.batches.append(lz.lz_batch_create(c.ctx, items, decompress=not want, stream=st))
            self.outs += [out, nb]

    @staticmethod
    def mix(requests):
        r = np.random.default_rng(requests)
        sym = r.choice([1, 2, 4], requests)
        sizes = np.minimum(r.lognormal(math.log(256 * KIB), 1.5, requests), 16 * MIB).astype(np.int64)
        comp = r.random(requests) < 0.7
        comp[0], comp[-1] = True, False
        return np.maximum(sizes // sym * sym, sym), sym, comp

    def run(self):
        c, st = _codec(), torch.cuda.current_stream().cuda_stream
        for b in self.batches:
            lz.lz_batch_run(c.ctx, b, st)
        return self.outs

    def __del__(self):
        st = torch.cuda.current_stream().cuda_stream
        for b in self.batches:
            lz.lz_batch_destroy(b, st)


# --- one pass ---------------------------------------------------------------------

def run(state):
    if isinstance(state, _Serve):
        return state.run()
    c, x, out, nb, op = (state[k] for k in ("codec", "x", "out", "nb", "op"))
    if op == "compress":
        return c.compress(x, state["p"], out=out, out_bytes=nb, **state["opt"])
    if op == "decompress":
        return c.decompress(x, n_bytes=state["n"], out=out, out_bytes=nb)
    st = torch.cuda.current_stream().cuda_stream
    if op == "host":
        size = lz.lz_compress_host(c.ctx, x.data_ptr(), x.numel(), state["p"], out.data_ptr(),
                                   out.numel(), st)
        return out, size
    fn = lz.lz_huff_compress if op == "huff_encode" else lz.lz_huff_decompress
    fn(c.ctx, x.data_ptr(), x.numel(), out.data_ptr(), out.numel(), nb.data_ptr(), st)
    return out, nb


def work(case):
    """Input read once, output written once (the stream's size from its usual
    share of the input); the codec does no floating-point work."""
    if case["op"] == "serve":
        sizes, sym, _ = _Serve.mix(case["requests"])
        share = np.array([STREAM_SHARE["markov%d" % (8 * s)] for s in sym])
        return {"bytes": int((sizes * (1 + share)).sum()), "flops": 0}
    share = HUFF_SHARE if case["op"].startswith("huff") else STREAM_SHARE
    return {"bytes": int(case["n"] * (1 + share[case["kind"]])), "flops": 0}
