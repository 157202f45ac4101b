"""Natural-order transforms of 64-bit words on both sides of the roomy limit
(2^48), at lengths of every kernel (short, whole rows, split with the order
written by the rows and by a pass of its own) and batches of one sequence and
of many: sampled outputs of Eq. 2 in Python integers, the round trip, and the
inputs whose lazy values are largest."""
import pytest
import torch

from gpu_util import need_gpu
from test_gpu_moduli64 import GENERAL, NEAR, ROOMY

pytestmark = pytest.mark.gpu

CASES = ([(ROOMY, L) for L in (0, 1, 3, 4, 7, 9, 10, 12, 13, 14, 15, 17)] + [(NEAR, 13)]
         + [(GENERAL, L) for L in (3, 9, 11, 13, 14, 15, 16)])


@pytest.mark.parametrize("m,L", CASES)
def test_transforms(m, L):
    need_gpu()
    from paper_1005_1497_gb300 import ntt
    N = 1 << L
    plan = ntt.Plan(m, N)
    order = 1                                                # of 2, a power of two
    while pow(2, order, m) != 1:
        order *= 2
    w = pow(2, order // N, m)
    gen = torch.Generator(device="cuda").manual_seed(L)
    for batch in (1, 40):
        x = torch.randint(0, m, (batch, N), generator=gen, dtype=torch.int64, device="cuda")
        x[0] = m - 1                                         # X(0) = -N, every other X(u) = 0
        x[-1, N // 2:] = 0
        X = ntt.ntt_forward(plan, x)
        assert torch.equal(ntt.ntt_inverse(plan, X), x), batch
        if batch > 1:
            want = torch.zeros(N, dtype=torch.int64)
            want[0] = (m - N) % m
            assert torch.equal(X[0].cpu(), want)
        row = x[-1].tolist()
        for u in {0, 1 % N, N // 2, N - 1, (5 * N) // 7}:
            step, p, s = pow(w, u, m), 1, 0
            for v in row[:max(1, N // 2)]:
                s = (s + v * p) % m
                p = p * step % m
            if N == 1:
                s = row[0]
            assert int(X[-1, u]) == s, (batch, u)
