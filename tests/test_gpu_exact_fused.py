"""The exact convolution's fused launches: one prime (the whole convolution in
one launch on the signed 64-bit inputs) and the second of two (the
reconstruction in its output), at every whole-sequence kernel's lengths,
batches of more than two rounds of the grid with a ragged end, bases that are
and are not 16-byte aligned, the output in place of an input; against the
separate passes word for word and against the oracle's exact convolution on
the first and last pairs."""
import math

import numpy as np
import pytest
import torch

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ntt():
    need_gpu()
    from paper_1005_1497_gb300 import ntt as mod
    mod.lib()
    return mod


def at(t, words):
    buf = torch.empty(t.numel() + words, dtype=t.dtype, device="cuda")
    out = buf[words:].view(t.shape)
    out.copy_(t)
    return out


def launches(ntt, plan, f, g, **kw):
    n = ntt.launch_count()
    h = ntt.conv_exact(plan, f, g, **kw)
    return h, ntt.launch_count() - n


# (log2 N, bound, primes, the override that selects the fused form)
CASES = ([(L, 22, 1, None) for L in (1, 2, 3, 5, 6, 8, 10, 11, 12, 13, 14)] + [(L, 40, 2, None) for L in (11, 12, 13)]
         + [(L, 40, 2, "1") for L in (6, 10)])


@pytest.mark.parametrize("L,bound,primes,override", CASES)
def test_fused_equals_passes_and_oracle(ntt, orc, monkeypatch, L, bound, primes, override):
    N = 1 << L
    monkeypatch.setenv("NTT_EXACT_FUSED", "0")
    passes = ntt.ExactPlan(N, bound)
    if override is None:
        monkeypatch.delenv("NTT_EXACT_FUSED")
    else:
        monkeypatch.setenv("NTT_EXACT_FUSED", override)
    plan = ntt.ExactPlan(N, bound)
    assert len(plan.primes) == primes and plan.primes == passes.primes
    amp = math.isqrt(((1 << bound) - 1) // N)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per_block = max(1, 512 * 32 >> max(L, 5))
    batch = 2 * sms * per_block + 1
    gen = torch.Generator(device="cuda").manual_seed(L)
    f, g = (torch.randint(-amp, amp + 1, (batch, N), generator=gen, device="cuda") for _ in range(2))
    f[0], g[0] = amp, -amp                                  # the extreme outputs of these amplitudes
    f[1], g[1] = -amp, -amp
    f[2], g[2] = 0, 0                                       # one input near the bound, far above 16 bits
    f[2, N - 1], g[2, 0] = -(1 << bound) + 1, 1
    want, separate = launches(ntt, passes, f, g)
    h, fused = launches(ntt, plan, f, g)
    assert fused < separate and fused * (primes + 2) == separate * (1 if primes == 1 else 3)
    assert torch.equal(h, want)
    for of, og, oh in ((1, 1, 1), (0, 1, 0), (1, 0, 1), (0, 0, 1)):
        out = at(torch.zeros_like(f), oh)
        assert torch.equal(ntt.conv_exact(plan, at(f, of), at(g, og), out=out), want), (of, og, oh)
    for words in (0, 1):
        x = at(f, words)
        assert torch.equal(ntt.conv_exact(plan, x, g, out=x), want)
    for b in (0, 1, 2, batch - 1):
        idx = np.unique(np.random.default_rng(L + b).integers(0, N, 64)).astype(np.uint64)
        got = want[b].cpu().numpy()[idx.astype(np.int64)]
        assert np.array_equal(got, orc.int_conv_sample(f[b].cpu().numpy(), g[b].cpu().numpy(), idx)), b
    plan.close()
    passes.close()


@pytest.mark.parametrize("L,bound,primes", [(L, 22, 1) for L in (2, 7, 12, 14)] + [(12, 40, 2)])
def test_inputs_of_the_whole_range(ntt, monkeypatch, L, bound, primes):
    """Any signed 64-bit input is reduced: beyond the plan's bound the outputs
    are the residues in (-M/2, M/2], the same words in both forms."""
    N = 1 << L
    monkeypatch.setenv("NTT_EXACT_FUSED", "0")
    passes = ntt.ExactPlan(N, bound)
    monkeypatch.setenv("NTT_EXACT_FUSED", "1")
    plan = ntt.ExactPlan(N, bound)
    assert len(plan.primes) == primes
    lo, hi = -(1 << 63), (1 << 63) - 1
    gen = torch.Generator(device="cuda").manual_seed(L)
    f, g = (torch.randint(lo, hi, (5, N), generator=gen, device="cuda") for _ in range(2))
    f[0], g[0] = lo, hi
    f[1], g[1] = lo, lo
    f[2], g[2] = -1, hi
    h = ntt.conv_exact(plan, f, g)
    assert torch.equal(h, ntt.conv_exact(passes, f, g))
    M = math.prod(plan.primes)
    h0 = N * lo * hi % M                                    # constant sequences: every output N lo hi
    assert h[0].cpu().tolist() == [h0 - M if h0 > (M - 1) // 2 else h0] * N
    plan.close()
    passes.close()
