"""The binding's buffer checks, without a GPU: an output (or work buffer) that
is too small, of another word size, strided, or in memory the GPU cannot
reach is rejected before the library is called, and one that fits -- exactly or with
room to spare -- is passed on."""
import ctypes
from types import SimpleNamespace

import pytest
import torch

from paper_1005_1497_gb300 import ntt

N = 16


class Buf:
    """What the binding looks at of a tensor."""

    def __init__(self, words, dtype=torch.int32, cuda=True, contiguous=True, shape=None):
        self.dtype, self.is_cuda, self._contiguous = dtype, cuda, contiguous
        self.shape = torch.Size(shape or (words,))
        self._words = words

    def numel(self):
        return self._words

    def element_size(self):
        return torch.empty(0, dtype=self.dtype).element_size()

    def is_contiguous(self):
        return self._contiguous

    def is_pinned(self):
        return False

    def data_ptr(self):
        return 4096


@pytest.fixture
def calls(monkeypatch):
    seen = []

    class Lib:
        def __getattr__(self, name):
            return lambda *args: seen.append(name) or 0
    monkeypatch.setattr(ntt, "lib", Lib)
    return seen


@pytest.fixture
def plan():
    p = ntt.Plan.__new__(ntt.Plan)
    p.handle, p.N, p.word_bits, p._dtypes = ctypes.c_void_p(), N, 32, (torch.int32, torch.uint32)
    return p


def entries(plan):
    """name -> call with the given output on two sequences of length N."""
    x, xe = Buf(2 * N), Buf(2 * N, torch.int64, shape=(2, N))
    exact = SimpleNamespace(handle=None, N=N)
    xs = Buf(2 * N, shape=(2, N))
    return {
        "ntt_forward": lambda o: ntt.ntt_forward(plan, x, o, stream=0),
        "ntt_inverse": lambda o: ntt.ntt_inverse(plan, x, o, stream=0),
        "conv_circular": lambda o: ntt.conv_circular(plan, x, x, o, stream=0),
        "conv_circular_noalloc": lambda o: ntt.conv_circular_noalloc(plan, x, x, o, stream=0),
        "conv_circular_plain": lambda o: ntt.conv_circular_plain(plan, x, x, o, Buf(4 * N), stream=0),
        "conv_circular_shift": lambda o: ntt.conv_circular_shift(641, xs, xs, o, stream=0),
        "conv_exact": lambda o: ntt.conv_exact(exact, xe, xe, o, stream=0),
    }


NAMES = ["ntt_forward", "ntt_inverse", "conv_circular", "conv_circular_noalloc", "conv_circular_plain",
         "conv_circular_shift", "conv_exact"]


@pytest.mark.parametrize("name", NAMES)
def test_output_that_does_not_fit_is_rejected(plan, calls, name):
    call = entries(plan)[name]
    exact = name == "conv_exact"
    dt, wrong = (torch.int64, torch.int32) if exact else (torch.int32, torch.int16)
    bad = [Buf(N, dt, shape=(1, N)), Buf(2 * N, wrong, shape=(2, N)), Buf(2 * N, dt, contiguous=False, shape=(2, N)),
           Buf(2 * N, dt, cuda=False, shape=(2, N))]
    for o in bad:
        with pytest.raises((ValueError, TypeError)):
            call(o)
    assert calls == []
    call(Buf(2 * N, dt, shape=(2, N)))
    assert calls == [name]


@pytest.mark.parametrize("name", ["ntt_forward", "ntt_inverse", "conv_circular", "conv_circular_plain", "conv_circular_shift"])
def test_output_with_room_to_spare_is_accepted(plan, calls, name):
    entries(plan)[name](Buf(3 * N))
    assert calls == [name]


def test_plain_work_buffer(plan, calls):
    x, out = Buf(2 * N), Buf(2 * N)
    for work in (Buf(4 * N - 1), Buf(4 * N, torch.int16), Buf(4 * N, cuda=False), Buf(4 * N, contiguous=False)):
        with pytest.raises(ValueError):
            ntt.conv_circular_plain(plan, x, x, out, work, stream=0)
    assert calls == []
    for work in (Buf(4 * N), Buf(4 * N, torch.float64)):
        ntt.conv_circular_plain(plan, x, x, out, work, stream=0)
    assert calls == ["conv_circular_plain"] * 2


@pytest.mark.parametrize("m,dtype,wrong", [(13631489, torch.int32, torch.int64), (70525124609, torch.int64, torch.int32)])
def test_batch_operands_of_another_word_size_are_rejected(calls, m, dtype, wrong):
    ok = Buf(N, dtype)
    for i in range(3):
        triple = [ok, ok, ok]
        triple[i] = Buf(N, wrong)
        for make in (ntt.conv_batched, ntt.BatchPlan):
            with pytest.raises(TypeError):
                make(m, [(ok, ok, ok), tuple(triple)])
    assert calls == []
    ntt.conv_batched(m, [(ok, ok, ok)], stream=0)
    assert calls == ["conv_batched"]


@pytest.mark.parametrize("m,dtype,wrong", [(13631489, torch.int32, torch.int16), (70525124609, torch.int64, torch.int32)])
def test_server_operands_that_do_not_fit_are_rejected(calls, m, dtype, wrong):
    srv = ntt.Server.__new__(ntt.Server)
    srv.handle, srv.m = ctypes.c_void_p(), m
    ok = Buf(N, dtype, cuda=False)
    bad = [Buf(N, wrong, cuda=False), Buf(N, dtype, cuda=False, contiguous=False)]
    for i in range(3):
        for b in bad + [Buf(N // 2, dtype, cuda=False)] * (i > 0):
            ops = [ok, ok, ok]
            ops[i] = b
            with pytest.raises((ValueError, TypeError)):
                srv.submit(*ops)
    assert calls == []
    srv.submit(ok, ok, ok)
    srv.submit(ok, Buf(2 * N, dtype), Buf(2 * N, dtype))
    assert calls == ["ntt_server_submit"] * 2


def test_range_check_of_another_word_size_is_rejected(plan, calls):
    for x in (Buf(N, torch.int16), Buf(N, torch.int64), Buf(N, contiguous=False), Buf(N, cuda=False)):
        with pytest.raises((ValueError, TypeError)):
            ntt.ntt_check_range(plan, x, stream=0)
    assert calls == []
    assert ntt.ntt_check_range(plan, Buf(N + 3), stream=0) == 0 and calls == ["ntt_check_range"]


def test_current_stream_without_the_raw_handle(monkeypatch):
    """A torch without the private calls that read the handle directly: the public one."""
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        monkeypatch.delattr(torch._C, name, raising=False)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=77))
    assert ntt._stream(None) == 77
