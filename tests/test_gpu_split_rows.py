"""The split path at every length and row length of its twist form: batches
of one pair, of one pair more than a wave of scratch, natural-order
transforms of the same plans, and rows whose last block is partly empty,
bit-exact against the row-twiddle form (itself pinned to the oracle) and the
round trip."""
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


@pytest.mark.parametrize("m,L", [(M, L) for L in range(15, 20)] + [(M64, L) for L in range(14, 21)])
def test_twist_rows_against_row_twiddles(ntt, monkeypatch, m, L):
    N = 1 << L
    monkeypatch.setenv("NTT_SPLIT_TWIST", "1")
    twist = ntt.Plan(m, N)
    monkeypatch.setenv("NTT_SPLIT_TWIST", "0")
    rows = ntt.Plan(m, N)
    assert twist.twist and not rows.twist
    gen = torch.Generator(device="cuda").manual_seed(L)
    for batch in (1, 3, 5):
        f = torch.randint(0, m, (batch, N), generator=gen, dtype=twist.dtype, device="cuda")
        g = torch.randint(0, m, (batch, N), generator=gen, dtype=twist.dtype, device="cuda")
        assert torch.equal(ntt.conv_circular(twist, f, g), ntt.conv_circular(rows, f, g)), batch
        X = ntt.ntt_forward(twist, f)
        assert torch.equal(X, ntt.ntt_forward(rows, f)), batch
        assert torch.equal(ntt.ntt_inverse(twist, X), f), batch
    top = torch.full((1, N), m - 1, dtype=twist.dtype, device="cuda")
    assert torch.equal(ntt.conv_circular(twist, top, top), torch.full_like(top, N % m))


@pytest.mark.parametrize("m,L", [(M, 15), (M, 17), (M64, 14), (M64, 16)])
def test_word_aligned_pointers(ntt, m, L):
    N = 1 << L
    plan = ntt.Plan(m, N)
    f, g = (dev(x, plan.word_bits) for x in pairs(m, 2, N, seed=70 + L))
    whole = ntt.conv_circular(plan, f, g)
    buf = [torch.empty(2 * N + 3, dtype=plan.dtype, device="cuda") for _ in range(3)]
    fs, gs, hs = (b[k:k + 2 * N].view(2, N) for b, k in zip(buf, (1, 2, 3)))
    fs.copy_(f)
    gs.copy_(g)
    assert torch.equal(ntt.conv_circular(plan, fs, gs, hs), whole)
    orc = oracle.Oracle()
    idx = np.random.default_rng(L).integers(0, N, 24, dtype=np.uint64)
    assert np.array_equal(host(whole)[1][idx.astype(np.int64)], orc.conv_sample(host(f)[1], host(g)[1], m, idx))


@pytest.mark.parametrize("m,L", [(M, 15), (M, 16), (M, 17), (M64, 14), (M64, 15)])
def test_natural_order_from_rows(ntt, monkeypatch, m, L):
    """Both sides of the tile limit above which the rows write the natural
    order, and more tiles than the grid holds, against the row-twiddle form."""
    N = 1 << L
    monkeypatch.setenv("NTT_SPLIT_TWIST", "1")
    twist = ntt.Plan(m, N)
    monkeypatch.setenv("NTT_SPLIT_TWIST", "0")
    rows = ntt.Plan(m, N)
    gen = torch.Generator(device="cuda").manual_seed(90 + L)
    for batch in (1, 2, 9, 40):
        f = torch.randint(0, m, (batch, N), generator=gen, dtype=twist.dtype, device="cuda")
        X = ntt.ntt_forward(rows, f)
        assert torch.equal(ntt.ntt_forward(twist, f), X), batch
        assert torch.equal(ntt.ntt_inverse(twist, X), f), batch
        y = f.clone()
        ntt.ntt_forward(twist, y, out=y)                      # in place
        assert torch.equal(y, X), batch
