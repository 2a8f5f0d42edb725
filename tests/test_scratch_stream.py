"""The hidden scratch of a chunked or paged call is taken in the order of the stream that the call is launched on: torch's allocator
hands a block that was freed on one stream out again to the same stream only."""
import contextlib

import pytest
import torch

from paper_2512_10411_b200 import binding


class _Stream:
    def __init__(self, cuda_stream):
        self.cuda_stream = cuda_stream


class _Foreign:  # a stream object of another library
    cuda_stream = 0x7700


CALLERS = 0x1100  # stands for the stream that is current where the call is made


class _Cuda(torch.Tensor):
    """A tensor in host memory that the binding takes for one on the GPU."""
    is_cuda = property(lambda self: True)
    device = property(lambda self: "cuda:0")


def _cuda(*shape, dtype=torch.bfloat16):
    return torch.zeros(shape, dtype=dtype).as_subclass(_Cuda)


class _Library:
    """Stand-in for libswaa: notes the scratch and the stream of each launch, and asks for `nbytes` of scratch."""

    def __init__(self, nbytes):
        self.nbytes, self.launches, self.asked = nbytes, [], 0

    def swaa_prefill_split_workspace_size(self, *args):
        self.asked += 1
        return self.nbytes

    def _split(self, *args):
        self.launches.append((args[-3], args[-1]))
        return 0

    def _plain(self, *args):
        self.launches.append((None, args[-1]))
        return 0

    swaa_prefill_chunked_split = swaa_prefill_paged_split = _split
    swaa_prefill_chunked = swaa_prefill_paged = swaa_prefill_chunked_mixed = swaa_prefill_paged_mixed = _plain


class _Block:
    def data_ptr(self):
        return 0xb10c

    def numel(self):
        return 4096


@pytest.fixture
def allocator(monkeypatch):
    """Stand-in for torch's streams and allocator: lists the streams that were current when memory was taken."""
    current, taken = [CALLERS], []

    @contextlib.contextmanager
    def stream_context(s):
        current.append(s.cuda_stream)
        try:
            yield
        finally:
            current.pop()

    def empty(nbytes, dtype, device):
        if nbytes > 1 << 30:
            raise torch.OutOfMemoryError("no memory left")
        taken.append((current[-1], nbytes, dtype, device))
        return _Block()

    monkeypatch.setattr(torch.cuda, "Stream", _Stream)
    monkeypatch.setattr(torch.cuda, "ExternalStream", lambda address, device=None: _Stream(address or 0xbad))  # 0 gives one from a pool
    monkeypatch.setattr(torch.cuda, "default_stream", lambda device=None: _Stream(0))
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: _Stream(current[-1]))
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: False)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    monkeypatch.setattr(torch.cuda, "stream", stream_context)
    return current, taken, empty


def _call(monkeypatch, allocator, nbytes, paged, stream):
    lib, lens = _Library(nbytes), torch.int32
    q, out, kv, cu = _cuda(3, 8, 128), _cuda(3, 8, 128), _cuda(6000, 2, 128), _cuda(4, dtype=lens)
    pages, table = _cuda(47, 128, 2, 128), _cuda(3, 47, dtype=lens)
    seqlens = _cuda(3, dtype=lens)
    with monkeypatch.context() as m:
        m.setattr(binding, "load_library", lambda: lib)
        m.setattr(torch, "empty", allocator[2])
        if paged:
            binding.swaa_prefill_paged(q, pages, pages, out, cu, seqlens, table, 1, 64, 4, True, stream=stream)
        else:
            binding.swaa_prefill_chunked(q, kv, kv, out, cu, cu, 1, 6000, 64, 4, True, stream=stream)
    return lib.launches


STREAMS = [(None, CALLERS), (_Stream(0x2200), 0x2200), (_Stream(0), 0), (0x3300, 0x3300), (0, 0), (_Foreign(), 0x7700)]


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("stream,launched_on", STREAMS)
def test_scratch_comes_from_the_launch_stream(monkeypatch, allocator, stream, launched_on, paged):
    current, taken, _ = allocator
    assert _call(monkeypatch, allocator, 4096, paged, stream) == [(0xb10c, launched_on)]
    assert taken == [(launched_on, 4096, torch.uint8, "cuda:0")]
    assert current == [CALLERS]


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("stream,launched_on", STREAMS)
def test_without_memory_the_call_goes_without_scratch(monkeypatch, allocator, stream, launched_on, paged):
    current, taken, _ = allocator
    assert _call(monkeypatch, allocator, 1 << 31, paged, stream) == [(None, launched_on)]
    assert taken == [] and current == [CALLERS]


@pytest.mark.parametrize("stream", [_Stream(0x2200), 0x3300, 0])
def test_while_the_callers_stream_is_captured_nothing_is_taken_for_another(monkeypatch, allocator, stream):
    _, taken, _ = allocator
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: True)
    assert _call(monkeypatch, allocator, 4096, False, stream) == [(None, getattr(stream, "cuda_stream", stream))]
    assert taken == []


@pytest.mark.parametrize("Tq,B,max_q,Hq,Hkv,asked", [
    (512, 1, 512, 8, 2, 0), (5, 1, 5, 8, 2, 0), (2, 1, 2, 8, 2, 1),    # one prompt; two tokens are eight rows
    (1024, 2, 512, 8, 2, 0), (515, 2, 512, 8, 2, 0), (514, 2, 512, 8, 2, 1),
    (520, 2, 512, 4, 4, 1), (521, 2, 512, 4, 4, 0), (100, 4, 50, 32, 2, 0), (100, 4, 50, 28, 4, 1),
])
def test_calls_without_room_for_a_generated_token_do_not_ask_for_scratch(monkeypatch, allocator, Tq, B, max_q, Hq, Hkv, asked):
    lib = _Library(4096)
    q, kv, cu = _cuda(Tq, Hq, 64), _cuda(3000, Hkv, 64), _cuda(B + 1, dtype=torch.int32)
    with monkeypatch.context() as m:
        m.setattr(binding, "load_library", lambda: lib)
        m.setattr(torch, "empty", allocator[2])
        binding.swaa_prefill_chunked(q, kv, kv, q, cu, cu, max_q, 3000, 64, 4, True)
    assert lib.asked == asked and lib.launches == [(0xb10c if asked else None, CALLERS)]
