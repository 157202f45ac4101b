"""The convolution by blocks at its edges: sequences whose addresses allow no
wide access (every pointer is aligned to the word only), every length from
the shortest that has blocks to the longest of one thread block, through the
contiguous and the descriptor form, and the largest moduli of both words
with every input m - 1 (the bounds' worst case: h = N mod m)."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import M, M64, dev, host, need_gpu, pairs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ntt():
    need_gpu()
    from paper_1005_1497_gb300 import ntt as mod
    mod.lib()
    return mod


@pytest.fixture(scope="module")
def orc():
    return oracle.Oracle()


def shifted(t, words):
    """A copy of t that starts `words` words after an allocation."""
    buf = torch.empty(t.numel() + words, dtype=t.dtype, device="cuda")
    out = buf[words:].view(t.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("m,L", [(M, L) for L in range(3, 15)] + [(M64, L) for L in range(3, 14)])
def test_word_aligned_pointers(ntt, orc, m, L):
    N = 1 << L
    plan = ntt.Plan(m, N)
    batch = plan.small_max + 5 if plan.small_max else 3      # past the one-block-per-pair limit
    f, g = pairs(m, batch, N, seed=4100 + L)
    w = orc.root(m, N)
    sample = sorted({0, 1, batch - 1})
    want = oracle.batched(lambda a, b: orc.fast_conv(a, b, m, w), f[sample], g[sample])
    fd, gd = dev(f, plan.word_bits), dev(g, plan.word_bits)
    whole = ntt.conv_circular(plan, fd, gd)
    assert np.array_equal(host(whole)[sample], want)
    for of, og, oh in ((1, 0, 0), (0, 1, 2), (3, 2, 1)):
        h = ntt.conv_circular(plan, shifted(fd, of), shifted(gd, og), shifted(torch.zeros_like(fd), oh))
        assert torch.equal(h, whole), (of, og, oh)
    triples = [(shifted(fd[b], b % 4), shifted(gd[b], (b + 1) % 4), shifted(torch.zeros_like(fd[b]), (b + 2) % 4))
               for b in range(min(batch, 7))]
    ntt.conv_batched(m, triples)
    torch.cuda.synchronize()
    for b, t in enumerate(triples):
        assert torch.equal(t[2], whole[b]), b


@pytest.mark.parametrize("m,L", [(26017793, 10), (26017793, 12), (26017793, 13), (59649589127497217, 4),
                                 (59649589127497217, 8), (1238926361552897, 9)])
def test_largest_moduli_worst_case(ntt, m, L):
    N = 1 << L
    plan = ntt.Plan(m, N)
    batch = plan.small_max + 3 if plan.small_max else 3
    f = torch.full((batch, N), m - 1, dtype=plan.dtype, device="cuda")
    assert torch.equal(ntt.conv_circular(plan, f, f), torch.full_like(f, N % m))
    assert torch.equal(ntt.conv_circular(plan, f[:1], f[:1]), torch.full_like(f[:1], N % m))
