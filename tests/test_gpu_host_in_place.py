"""Page-locked host buffers that the kernels read in place: the lengths with
kernels of their own for it, batches above and below one block per pair,
addresses that allow 16-byte, 8-byte and single-word accesses, bit-exact
against the device call."""
import pytest
import torch

from gpu_util import M, M64, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,L", [(M, L) for L in range(9, 15)] + [(M64, 9), (M64, 13)])
def test_in_place(m, L):
    need_gpu()
    from paper_1005_1497_gb300 import ntt
    N = 1 << L
    plan = ntt.Plan(m, N)
    gen = torch.Generator(device="cuda").manual_seed(L)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for batch in (1, 2 * sms + 1):
        f, g = (torch.randint(0, m, (batch, N), generator=gen, dtype=plan.dtype, device="cuda") for _ in range(2))
        want = ntt.conv_circular(plan, f, g).cpu()
        for offs in ((0, 0, 0), (2, 2, 2), (1, 2, 3)):
            bufs = [torch.full((batch * N + 4,), -1, dtype=plan.dtype, pin_memory=True) for _ in range(3)]
            fh, gh, hh = (b[o:o + batch * N].view(batch, N) for b, o in zip(bufs, offs))
            fh.copy_(f)
            gh.copy_(g)
            ntt.conv_circular_host(plan, fh, gh, hh)
            assert torch.equal(hh, want), (batch, offs)
            o = offs[2]
            assert bool((bufs[2][:o] == -1).all()) and bool((bufs[2][o + batch * N:] == -1).all())
