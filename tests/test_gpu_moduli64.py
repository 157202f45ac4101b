"""64-bit words on both sides of the roomy limit (2^48): Rader primes close
below it and above it, at lengths of every kernel (short, column/row, split
with one column pass), against sampled outputs of
Eq. 1, and with every input m - 1, where h = N mod m and the lazy values are
largest."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import dev, host, need_gpu, pairs

pytestmark = pytest.mark.gpu

NEAR = 151413703311361        # a factor of F_27, 2^47.1 (its order of 2, 2^28, makes plans slow: two lengths)
ROOMY = 31065037602817        # a factor of F_17, 2^44.8: N up to 2^18
GENERAL = 2327042503868417    # a factor of F_15, 2^51.05: N up to 2^16
CASES = ([(ROOMY, L) for L in (1, 2, 3, 5, 8, 9, 10, 12, 13, 14, 16, 18)] + [(NEAR, L) for L in (9, 13)]
         + [(GENERAL, L) for L in (1, 2, 3, 5, 8, 9, 10, 11, 12, 13, 14, 15, 16)])


@pytest.fixture(scope="module")
def ntt():
    need_gpu()
    from paper_1005_1497_gb300 import ntt as mod
    mod.lib()
    return mod


@pytest.mark.parametrize("m,L", CASES)
def test_both_sides_of_the_roomy_limit(ntt, m, L):
    N = 1 << L
    plan = ntt.Plan(m, N)
    assert plan.word_bits == 64
    batch = plan.small_max + 2 if plan.small_max else 2
    f, g = pairs(m, batch, N, seed=500 + L)
    h = ntt.conv_circular(plan, dev(f, 64), dev(g, 64))
    orc = oracle.Oracle()
    idx = np.random.default_rng(L).integers(0, N, min(N, 32), dtype=np.uint64)
    for b in (0, batch - 1):
        assert np.array_equal(host(h[b])[idx.astype(np.int64)], orc.conv_sample(f[b], g[b], m, idx)), b
    triples = [(dev(f[b], 64), dev(g[b], 64), torch.empty(N, dtype=torch.int64, device="cuda")) for b in range(2)]
    ntt.conv_batched(m, triples)
    torch.cuda.synchronize()
    assert all(torch.equal(t[2], h[b]) for b, t in enumerate(triples))
    top = torch.full((batch, N), m - 1, dtype=torch.int64, device="cuda")
    assert torch.equal(ntt.conv_circular(plan, top, top), torch.full_like(top, N % m))
