"""Uneven batches of 64-bit words on both sides of the roomy limit (2^48), with
more pairs per length than two rounds of a block of the persistent launch and
a ragged end, against the uniform convolution (which the oracle checks)."""
import pytest
import torch

from gpu_util import M64, need_gpu

pytestmark = pytest.mark.gpu

GENERAL = 2327042503868417    # a factor of F_15, 2^51.05: N up to 2^16


@pytest.mark.parametrize("m", [M64, GENERAL])
def test_uneven_batch(m):
    need_gpu()
    from paper_1005_1497_gb300 import ntt
    gen = torch.Generator(device="cuda").manual_seed(7)
    triples, want = [], []
    for L in (1, 3, 5, 6, 7, 8, 9, 10, 12, 13, 14, 15):
        N = 1 << L
        count = max(3, 4 * (512 * 16 >> max(L, 4)) + 1)
        f, g = (torch.randint(0, m, (count, N), generator=gen, dtype=torch.int64, device="cuda") for _ in range(2))
        h = torch.full((count, N), -1, dtype=torch.int64, device="cuda")
        want.append((h, ntt.conv_circular(ntt.Plan(m, N), f, g)))
        triples += [(f[b], g[b], h[b]) for b in range(count)]
    batch = ntt.BatchPlan(m, triples)
    batch.exec()
    for h, w in want:
        assert torch.equal(h, w), h.shape
        h.fill_(-1)
    batch.exec_graph()
    for h, w in want:
        assert torch.equal(h, w), h.shape
    batch.close()
