"""Natural-order transforms of the lengths that one thread holds (reordered in
registers, 16-byte accesses where a sequence is aligned) and of those whose
rows share a warp: every offset of input and output from a 16-byte boundary,
in place, batches of one sequence and of more than two rounds of the grid
with a ragged end, against the oracle, and nothing written beside the
output."""
import numpy as np
import pytest
import torch

from gpu_util import M, M64, host, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,L", [(M, L) for L in range(10)] + [(M64, L) for L in range(9)])
def test_offsets_and_batches(orc, m, L):
    need_gpu()
    from paper_1005_1497_gb300 import ntt
    N = 1 << L
    plan = ntt.Plan(m, N)
    word = plan.word_bits
    steps = 16 * 8 // word                                  # offsets in words
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per_block = 512 if N * word <= 1024 else 512 * 1024 // (N * word)
    gen = torch.Generator(device="cuda").manual_seed(L)
    for batch in (1, 2 * sms * per_block + 1):
        x = torch.randint(0, m, (batch, N), generator=gen, dtype=plan.dtype, device="cuda")
        for inverse in (False, True):
            run = ntt.ntt_inverse if inverse else ntt.ntt_forward
            want = run(plan, x)
            for b in {0, batch // 2, batch - 1}:
                row = host(x[b])
                X = orc.ntt(row, m, plan.omega)
                if inverse:                                 # N^-1 F at <-u>_N
                    ninv = pow(N, -1, m)
                    X = np.array([int(X[-u % N]) * ninv % m for u in range(N)], dtype=np.uint64)
                assert np.array_equal(host(want[b]), X), (inverse, b)
            for i in range(steps):
                for o in range(steps):
                    xb = torch.empty(batch * N + steps, dtype=x.dtype, device="cuda")
                    yb = torch.full((batch * N + 2 * steps,), -1, dtype=x.dtype, device="cuda")
                    xi, yo = xb[i:i + batch * N].view(batch, N), yb[o:o + batch * N].view(batch, N)
                    xi.copy_(x)
                    run(plan, xi, yo)
                    assert torch.equal(yo, want), (inverse, i, o)
                    assert bool((yb[:o] == -1).all()) and bool((yb[o + batch * N:] == -1).all())
                    run(plan, xi, xi)
                    assert torch.equal(xi, want), (inverse, i)
