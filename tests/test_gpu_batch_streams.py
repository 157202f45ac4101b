"""Batch plans whose classes run on one, two and three streams and share
scratch there: work-list lengths alone, one class of at most a round, many
such classes (split ones among them) beside a class that fills the GPU, and a
split class of more pairs than one wave of scratch, bit-exact against the
contiguous call of every length, directly and by graph replay."""
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


CLASSES = [                                                  # (modulus, {log2 N: pairs})
    (M, {6: 5, 3: 2}),
    (M, {13: 1}),
    (M, {16: 3}),
    (M, {17: 3, 15: 9, 19: 1, 16: 2}),
    (M, {7: 40, 11: 30, 12: 3, 13: 20, 14: 400, 15: 200, 16: 5, 18: 1}),
    (M, {17: 1100, 15: 3}),
    (M64, {5: 9, 9: 3, 12: 4, 13: 350, 14: 6, 17: 2}),
]


@pytest.mark.parametrize("m,classes", CLASSES)
def test_classes_on_streams(ntt, m, classes):
    gen = torch.Generator(device="cuda").manual_seed(len(classes))
    want, triples, outs = [], [], []
    for L, count in classes.items():
        plan = ntt.Plan(m, 1 << L)
        f, g = (torch.randint(0, m, (count, 1 << L), generator=gen, dtype=plan.dtype, device="cuda") for _ in range(2))
        h = torch.empty_like(f)
        want.append(ntt.conv_circular(plan, f, g))
        outs.append(h)
        triples += [(f[i], g[i], h[i]) for i in range(count)]
    order = torch.randperm(len(triples), generator=torch.Generator().manual_seed(1)).tolist()
    batch = ntt.BatchPlan(m, [triples[i] for i in order])
    for run in (batch.exec, batch.exec_graph, batch.exec_graph):
        for h in outs:
            h.fill_(-1)
        run()
        for h, w in zip(outs, want):
            assert torch.equal(h, w)
    batch.close()
