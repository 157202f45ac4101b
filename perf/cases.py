"""The library's work as its users have it done, as measurable cases.

Each case goes through the Python binding's public entry points on random
residues (the only data the method knows: every word uniform in [0, m)).
Sizes are those of the benchmark's workloads and of the tests, and others of
the same ranges.  `listed()` has the fixed cases, `draw()` more of the same
kinds; `exact()` recomputes a case's result in 64-bit integers (doubles for
the integer convolution, whose values they hold exactly) with plain torch.

Kinds:
  conv      conv_circular on a contiguous batch of device pairs
  forward   ntt_forward, natural order
  inverse   ntt_inverse, natural order
  uneven    a batch plan of pairs of many lengths, replayed as a CUDA graph
  exact     conv_exact, signed integers without a modulus
  shift     conv_circular_shift, the strict bit-shift form
  host      conv_circular_host, page-locked host buffers in and out
"""
from __future__ import annotations

import math
import random

import torch

from paper_1005_1497_gb300 import inputs, ntt

M32 = 13631489           # factor of F_18: 32-bit words, every length up to 2^19
M64 = 70525124609        # factor of F_19: 64-bit words, every length up to 2^20
SMALL = {641: 64, 65537: 32, 6700417: 64}      # factors of F_5 and F_4: the largest length of the shift form


def listed():
    return [
        # one filter call on one short signal: latency, a single launch
        {"name": "conv_single_1k", "kind": "conv", "m": M32, "log2n": 10, "batch": 1},
        # very many short blocks (block-wise filtering), a ragged count
        {"name": "conv_short_256", "kind": "conv", "m": M32, "log2n": 8, "batch": 20011},
        # the uniform batch, the library's headline workload
        {"name": "conv_batch_16k", "kind": "conv", "m": M32, "log2n": 14, "batch": 4096},
        # the longest 32-bit-word transforms: the split path
        {"name": "conv_large_512k", "kind": "conv", "m": M32, "log2n": 19, "batch": 64},
        # 64-bit words at the serving mix's median length, an odd batch
        {"name": "conv64_8k", "kind": "conv", "m": M64, "log2n": 13, "batch": 301},
        # 64-bit words on the split path
        {"name": "conv64_128k", "kind": "conv", "m": M64, "log2n": 17, "batch": 12},
        # spectra of a batch of signals, whole sequences
        {"name": "forward_16k", "kind": "forward", "m": M32, "log2n": 14, "batch": 4096},
        # signals back from longer spectra, split path, a ragged batch
        {"name": "inverse_64k", "kind": "inverse", "m": M32, "log2n": 16, "batch": 333},
        # a batch of uneven lengths planned once and replayed
        {"name": "uneven_2000", "kind": "uneven", "m": M32, "lo": 6, "hi": 19, "count": 2000, "mix": 3},
        # exact integer filtering of 16-bit samples (two primes, Chinese remainder theorem)
        {"name": "exact_4k", "kind": "exact", "log2n": 12, "batch": 5001, "bits": 16},
        # many tiny convolutions in the literal bit-shift form
        {"name": "shift_64", "kind": "shift", "m": 641, "log2n": 6, "batch": 1000003},
        # a batch whose signals live in page-locked host memory
        {"name": "host_16k", "kind": "host", "m": M32, "log2n": 14, "batch": 600},
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["conv", "conv", "conv", "conv64", "conv64", "forward", "inverse", "uneven", "exact", "shift", "host"])
    if kind == "conv":
        k = rng.randint(6, 19)
        return {"kind": "conv", "m": M32, "log2n": k, "batch": _log_int(rng, 1, (1 << 25) >> k)}
    if kind == "conv64":
        k = rng.randint(6, 18)
        return {"kind": "conv", "m": M64, "log2n": k, "batch": _log_int(rng, 1, (1 << 22) >> k)}
    if kind in ("forward", "inverse"):
        m = rng.choice([M32, M32, M64])
        k = rng.randint(8, 18)
        return {"kind": kind, "m": m, "log2n": k, "batch": _log_int(rng, 1, (1 << (25 if m == M32 else 23)) >> k)}
    if kind == "uneven":
        return {"kind": "uneven", "m": M32, "lo": 6, "hi": rng.randint(12, 19), "count": _log_int(rng, 50, 1500),
                "mix": rng.randint(0, 1 << 20)}
    if kind == "exact":
        k, bits = rng.randint(8, 16), rng.choice([12, 14, 16])
        return {"kind": "exact", "log2n": k, "batch": _log_int(rng, 1, (1 << 24) >> k), "bits": bits}
    if kind == "shift":
        m = rng.choice(sorted(SMALL))
        k = rng.randint(2, 5 if m == 65537 else 6)
        return {"kind": "shift", "m": m, "log2n": k, "batch": _log_int(rng, 1000, (1 << 26) >> k)}
    k = rng.randint(10, 16)
    return {"kind": "host", "m": M32, "log2n": k, "batch": _log_int(rng, 1, (1 << 23) >> k)}


# ------------------------------------------------------------------- inputs

def _words(m: int) -> torch.dtype:
    return torch.int32 if m < (1 << 25) else torch.int64


def _lengths(case):
    """The lengths of an uneven batch: part of the case, not of its inputs."""
    return inputs.log_uniform_lengths(case["count"], case["lo"], case["hi"], seed=case["mix"]).tolist()


def _random(case, seed):
    """The case's input tensors on the GPU, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "exact":
        shape, half = (case["batch"], 1 << case["log2n"]), 1 << (case["bits"] - 1)
        return [torch.randint(-half, half, shape, generator=gen, dtype=torch.int64, device="cuda") for _ in range(2)]
    m = case["m"]
    shape = (sum(_lengths(case)),) if kind == "uneven" else (case["batch"], 1 << case["log2n"])
    count = 1 if kind in ("forward", "inverse") else 2
    return [torch.randint(0, m, shape, generator=gen, dtype=_words(m), device="cuda") for _ in range(count)]


def prepare(case, seed):
    kind, x = case["kind"], _random(case, seed)
    st = {"case": case, "x": x}
    if kind in ("conv", "forward", "inverse"):
        st["plan"] = ntt.Plan(case["m"], 1 << case["log2n"])
    elif kind == "exact":
        st["plan"] = ntt.ExactPlan(1 << case["log2n"], case["log2n"] + 2 * case["bits"])
    elif kind == "host":
        st["plan"] = ntt.Plan(case["m"], 1 << case["log2n"])
        st["x"] = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in x]
        st["h"] = torch.empty(x[0].shape, dtype=x[0].dtype, pin_memory=True)
    elif kind == "uneven":
        f, g = x
        st["h"] = torch.empty_like(f)
        triples, at = [], 0
        for n in _lengths(case):
            triples.append((f[at:at + n], g[at:at + n], st["h"][at:at + n]))
            at += n
        st["plan"] = ntt.BatchPlan(case["m"], triples)
    return st


def run(st):
    case, x = st["case"], st["x"]
    kind = case["kind"]
    if kind == "conv":
        return ntt.conv_circular(st["plan"], x[0], x[1])
    if kind == "forward":
        return ntt.ntt_forward(st["plan"], x[0])
    if kind == "inverse":
        return ntt.ntt_inverse(st["plan"], x[0])
    if kind == "exact":
        return ntt.conv_exact(st["plan"], x[0], x[1])
    if kind == "shift":
        return ntt.conv_circular_shift(case["m"], x[0], x[1])
    if kind == "host":
        return ntt.conv_circular_host(st["plan"], x[0], x[1], st["h"])
    st["plan"].exec_graph()
    return st["h"]


def work(case):
    """Bytes: each input word read once, each output word written once.
    Flops: a multiplication and an addition for each modular product of the
    radix-2 transforms and the pointwise product (per prime where the integer
    convolution needs two)."""
    kind = case["kind"]
    if kind == "uneven":
        lens = _lengths(case)
        return {"bytes": 12 * sum(lens), "flops": 2 * sum(3 * n // 2 * (n.bit_length() - 1) + n for n in lens)}
    k, total = case["log2n"], case["batch"] << case["log2n"]
    if kind == "exact":
        return {"bytes": 24 * total, "flops": 2 * 2 * total * (3 * k / 2 + 1)}
    size = 4 if case["m"] < (1 << 25) else 8
    if kind in ("forward", "inverse"):
        return {"bytes": 2 * size * total, "flops": 2 * total * k / 2}
    return {"bytes": 3 * size * total, "flops": 2 * total * (3 * k / 2 + 1)}


# ---------------------------------------------------------- 64-bit recomputation

def _mul(a, b, m):
    """a b mod m for residues below 2^37, in 64-bit integers."""
    if m < (1 << 31):
        return a * b % m
    return ((a * (b >> 18) % m << 18) + a * (b & 0x3FFFF)) % m


def _root(m, n):
    """2^(ord/n) mod m, ord the (power-of-two) order of 2."""
    order = 1
    while pow(2, order, m) != 1:
        order *= 2
    return pow(2, order // n, m)


def _powers(w, count, m, device):
    p, step = torch.ones(1, dtype=torch.int64, device=device), w
    while p.numel() < count:
        p = torch.cat([p, _mul(p, torch.full_like(p, step), m)])
        step = step * step % m
    return p


def _transform(x, w, m):
    """Radix-2 decimation in frequency; natural order in and out."""
    n = x.shape[-1]
    y, h, pw = x, n // 2, _powers(w, max(1, n // 2), m, x.device)
    while h >= 1:
        v = y.reshape(-1, n // (2 * h), 2, h)
        a, b = v[:, :, 0], v[:, :, 1]
        y = torch.stack([(a + b) % m, _mul((a - b) % m, pw[::n // (2 * h)], m)], dim=2).reshape(-1, n)
        h //= 2
    k = n.bit_length() - 1
    i = torch.arange(n, device=x.device)
    r = torch.zeros_like(i)
    for s in range(k):
        r |= (i >> s & 1) << (k - 1 - s)
    return y[:, r]


def _conv(f, g, m):
    n = f.shape[-1]
    w = _root(m, n)
    h = _mul(_transform(f, w, m), _transform(g, w, m), m)
    h = _transform(h, pow(w, -1, m), m)
    return _mul(h, torch.full_like(h, pow(n, -1, m)), m)


def exact(case, seed):
    kind, x = case["kind"], [t.to(torch.int64) for t in _random(case, seed)]
    if kind == "exact":
        out = [torch.fft.irfft(torch.fft.rfft(f.double()) * torch.fft.rfft(g.double()), n=1 << case["log2n"])
               for f, g in zip(x[0].split(512), x[1].split(512))]
        return torch.cat(out).round().to(torch.int64)
    m = case["m"]
    if kind in ("forward", "inverse"):
        n = 1 << case["log2n"]
        w = _root(m, n)
        y = _transform(x[0], w if kind == "forward" else pow(w, -1, m), m)
        if kind == "inverse":
            y = _mul(y, torch.full_like(y, pow(n, -1, m)), m)
        return y.to(_words(m))
    if kind == "shift":
        n = 1 << case["log2n"]
        h = torch.zeros_like(x[0])
        for k in range(n):
            h += x[0][:, k:k + 1] * torch.roll(x[1], k, dims=1)
        return (h % m).to(torch.int32)
    if kind == "uneven":
        lens = _lengths(case)
        h, at, where = torch.empty_like(x[0]), 0, {}
        for n in lens:
            where.setdefault(n, []).append(at)
            at += n
        for n, starts in where.items():
            for some in [starts[i:i + 64] for i in range(0, len(starts), 64)]:
                idx = torch.tensor(some, device=h.device)[:, None] + torch.arange(n, device=h.device)
                h[idx] = _conv(x[0][idx], x[1][idx], m)
        return h.to(torch.int32)
    h = torch.cat([_conv(f, g, m) for f, g in zip(x[0].split(1024), x[1].split(1024))]).to(_words(m))
    return h.cpu() if kind == "host" else h
