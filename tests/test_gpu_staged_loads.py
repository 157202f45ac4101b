"""Kernels that stage their next sequence by asynchronous copies: batches of
one group, one block and more than one round of the grid with a ragged end,
with addresses that allow 16-byte copies, 8-byte copies and only single
words, natural-order transforms and short convolutions."""
import pytest
import torch

from gpu_util import M, M64, need_gpu

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


@pytest.mark.parametrize("m,L", [(M, L) for L in (0, 1, 3, 5, 6, 7, 8, 9, 10, 11, 13, 14)] + [(M64, L) for L in (0, 2, 4, 5, 6, 8, 9, 10, 13)])
def test_batches_and_alignments(ntt, m, L):
    N = 1 << L
    plan = ntt.Plan(m, N)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per_block = max(1, (512 << (5 if m == M else 4)) >> L) if L > (5 if m == M else 4) else 512
    gen = torch.Generator(device="cuda").manual_seed(L)
    for batch in (1, per_block + 1, 2 * sms * per_block + 1):
        x = torch.randint(0, m, (batch, N), generator=gen, dtype=plan.dtype, device="cuda")
        y = torch.randint(0, m, (batch, N), generator=gen, dtype=plan.dtype, device="cuda")
        X = ntt.ntt_forward(plan, x)
        assert torch.equal(ntt.ntt_inverse(plan, X), x), batch
        h = ntt.conv_circular(plan, x, y)
        for w in (1, 2, 3):
            assert torch.equal(ntt.ntt_forward(plan, at(x, w)), X), (batch, w)
            assert torch.equal(ntt.conv_circular(plan, at(x, w), at(y, 3 - w)), h), (batch, w)
        # the convolution theorem on a few pairs ties the three results together
        if m == M:
            G = ntt.ntt_forward(plan, y[:3].contiguous())
            prod = (X[:3].to(torch.int64) * G.to(torch.int64) % m).to(plan.dtype)
            assert torch.equal(ntt.ntt_inverse(plan, prod), h[:3]), batch
