"""The shift kernel's two register passes at the edges of its mapping: one
pair, one more or less than a block's pairs, more pairs than the grid holds
at once, and the values at which its lazy words are largest (all m - 1, and
impulses of m - 1 that reach every output), in both modes, against the main
path (itself bit-exact against the oracle)."""
import pytest
import torch

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

CASES = [(641, 6), (6700417, 6), (6700417, 5), (641, 4), (65537, 5), (65537, 4), (65537, 3), (641, 3), (641, 2), (65537, 1)]


@pytest.fixture(scope="module")
def ntt():
    need_gpu()
    from paper_1005_1497_gb300 import ntt as mod
    mod.lib()
    return mod


@pytest.mark.parametrize("m,L", CASES)
def test_shift_batches_and_extremes(ntt, m, L):
    N = 1 << L
    plan = ntt.Plan(m, N)
    block = 256 // max(1, N // 8)                              # pairs of one block
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    gen = torch.Generator(device="cuda").manual_seed(7 * L + m)
    for batch in (1, block - 1, block + 1, 8 * sms * block + 1):
        f = torch.randint(0, m, (batch, N), generator=gen, dtype=torch.int32, device="cuda")
        g = torch.randint(0, m, (batch, N), generator=gen, dtype=torch.int32, device="cuda")
        want = ntt.conv_circular(plan, f, g)
        for mode in (ntt.SHIFT_STRICT, ntt.SHIFT_SHOUP):
            assert torch.equal(ntt.conv_circular_shift(m, f, g, mode=mode), want), (batch, mode)
    eye = torch.eye(N, dtype=torch.int32, device="cuda") * (m - 1)
    top = torch.full((N, N), m - 1, dtype=torch.int32, device="cuda")
    for f, g in ((eye, top), (top, top), (eye, eye)):
        want = ntt.conv_circular(plan, f, g)
        for mode in (ntt.SHIFT_STRICT, ntt.SHIFT_SHOUP):
            assert torch.equal(ntt.conv_circular_shift(m, f, g, mode=mode), want), mode
