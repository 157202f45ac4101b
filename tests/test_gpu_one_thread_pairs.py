"""Convolutions of the lengths that one thread holds (16-byte accesses where a
sequence is aligned): batch plans whose f, g and h lie at every offset from a
16-byte boundary, beside a longer length in the same persistent launch,
against the oracle, and nothing written beside the outputs."""
import numpy as np
import pytest
import torch

from gpu_util import M, M64, dev, host, need_gpu, pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,lengths", [(M, (1, 2, 3, 4, 5, 10)), (M64, (1, 2, 3, 4, 9))])
def test_offsets_from_16_bytes(orc, m, lengths):
    need_gpu()
    from paper_1005_1497_gb300 import ntt
    word = 32 if m == M else 64
    steps = 16 * 8 // word                                  # offsets in words
    offsets = [(a, b, c) for a in range(steps) for b in range(steps) for c in range(steps)]
    triples, checks = [], []
    for L in lengths:
        N = 1 << L
        f, g = pairs(m, len(offsets), N, seed=900 + L)
        fd, gd = dev(f, word), dev(g, word)
        size = 2 * max(N, steps) + steps                    # a multiple of 16 bytes, with room around the sequence
        bufs = [torch.full((len(offsets), size), -1, dtype=fd.dtype, device="cuda") for _ in range(3)]
        for i, (a, b, c) in enumerate(offsets):
            ft, gt, ht = (buf[i, steps + o:steps + o + N] for buf, o in zip(bufs, (a, b, c)))
            ft.copy_(fd[i])
            gt.copy_(gd[i])
            triples.append((ft, gt, ht))
        checks.append((L, f, g, bufs[2]))
    plan = ntt.BatchPlan(m, triples)
    plan.exec()
    torch.cuda.synchronize()
    for L, f, g, hb in checks:
        N = 1 << L
        for i, (_, _, c) in enumerate(offsets):
            at = steps + c
            assert np.array_equal(host(hb[i, at:at + N]), orc.conv(f[i], g[i], m)), (L, i)
            assert bool((hb[i, :at] == -1).all()) and bool((hb[i, at + N:] == -1).all()), (L, i)
    plan.close()
