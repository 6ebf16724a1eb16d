"""Scratch that the binding provides: calls into other streams than the current one, and into streams that are being captured."""
import ctypes as C
import gc

import pytest
import torch

from _routes import Streaming

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def e3():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2505_18573_b200 import binding
    binding.lib()
    return Streaming(binding)  # (the kernel of short calls has no use for scratch)


class _Calls:
    """A sampling call with outputs of its own; rows few enough to be cut, so that the scratch is written."""

    def __init__(self, e3, rows=5, V=50000):
        g = torch.Generator(device=DEV); g.manual_seed(rows)
        self.e3, self.logits = e3, torch.randn((rows, V), generator=g, device=DEV)
        self.temps = torch.full((rows,), 0.8, device=DEV)
        self.tok = torch.empty(rows, dtype=torch.int32, device=DEV)
        self.logp, self.ent = torch.empty(rows, device=DEV), torch.empty(rows, device=DEV)
        self.need = e3.e3_workspace_bytes(e3.E3_CALL_SAMPLE, rows, V, e3.E3_F32)

    def __call__(self, stream):
        self.e3.e3_sample(self.logits, self.temps, 3, 4, sampler=self.e3.E3_SAMPLER_BLOCK, out_tok=self.tok, out_logp=self.logp, out_ent=self.ent, stream=stream)

    def results(self):
        torch.cuda.synchronize()
        return self.tok.clone(), self.logp.clone(), self.ent.clone()

    def clear(self):
        self.tok.fill_(-7); self.logp.zero_(); self.ent.zero_()


def test_the_calls_here_write_their_scratch(e3):
    for calls in (_Calls(e3), _Calls(e3, 3), _Calls(e3, 8), _Calls(e3, 40, 150000), _Calls(e3, 700)):
        room = torch.full((calls.need,), 0x5A, dtype=torch.uint8, device=DEV)
        e3.e3_sample(calls.logits, calls.temps, 3, 4, sampler=e3.E3_SAMPLER_BLOCK, workspace=room)
        assert bool((room != 0x5A).any())


def _canaries(stream, nbytes):
    """Memory that torch has free for `stream` and for the current one, filled with a pattern."""
    out = []
    for s in (stream, torch.cuda.current_stream()):
        with torch.cuda.stream(s):
            out += [torch.full((nbytes,), 0x5A, dtype=torch.uint8, device=DEV) for _ in range(4)]
    torch.cuda.synchronize()
    return out


def _replay_touches_only_its_own(e3, calls, want, replay, stream):
    big = _Calls(e3, 700, 50000)  # outgrows the buffer that is kept for the stream
    big(stream)
    torch.cuda.synchronize()
    held = _canaries(stream, calls.need)
    for _ in range(3):
        calls.clear()
        torch.cuda.synchronize()
        replay()
        assert all(torch.equal(a, b) for a, b in zip(want, calls.results()))
        assert all(bool((t == 0x5A).all()) for t in held)


def test_capture_of_a_stream_that_is_not_current(e3):
    calls, side = _Calls(e3), torch.cuda.Stream()
    calls(side)
    want = calls.results()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        side.wait_stream(torch.cuda.current_stream())
        calls(side)
        beside = torch.full((calls.need,), 0x5A, dtype=torch.uint8, device=DEV)  # (not ordered with the call)
        torch.cuda.current_stream().wait_stream(side)
    _replay_touches_only_its_own(e3, calls, want, graph.replay, side)
    assert bool((beside == 0x5A).all())


def _runtime():
    lib = C.CDLL("libcudart.so.12")

    def call(name, *args):
        assert getattr(lib, name)(*args) == 0, name
    return call


@pytest.mark.parametrize("current", [True, False])
def test_capture_without_torch(e3, current):
    """A capture that torch does not know of: the scratch belongs to the graph, not to torch's free memory."""
    calls, side, call = _Calls(e3, 6), torch.cuda.Stream(), _runtime()
    calls(side)
    want = calls.results()
    handle, graph, runnable = C.c_void_p(side.cuda_stream), C.c_void_p(), C.c_void_p()
    call("cudaStreamBeginCapture", handle, 1)  # thread-local
    with torch.cuda.stream(side if current else torch.cuda.current_stream()):
        calls(side)
        calls(side)  # (the same buffer)
    call("cudaStreamEndCapture", handle, C.byref(graph))
    call("cudaGraphInstantiate", C.byref(runnable), graph, C.c_ulonglong(0))
    call("cudaGraphDestroy", graph)
    _replay_touches_only_its_own(e3, calls, want, lambda: call("cudaGraphLaunch", runnable, handle), side)
    torch.cuda.synchronize()
    call("cudaGraphExecDestroy", runnable)


def test_memory_of_dropped_graphs_comes_back(e3):
    calls, side, call = _Calls(e3, 40, 150000), torch.cuda.Stream(), _runtime()
    calls(side)
    torch.cuda.synchronize()
    gc.collect()
    base = torch.cuda.memory_allocated()
    handle = C.c_void_p(side.cuda_stream)
    for _ in range(20):
        graph = C.c_void_p()
        call("cudaStreamBeginCapture", handle, 1)
        calls(side)
        call("cudaStreamEndCapture", handle, C.byref(graph))
        call("cudaGraphDestroy", graph)
        torch.cuda.synchronize()
    import time
    for _ in range(100):  # (given back on a thread of the runtime, then by the next call)
        calls(side)
        torch.cuda.synchronize()
        if torch.cuda.memory_allocated() <= base:
            break
        time.sleep(0.02)
    assert torch.cuda.memory_allocated() <= base


def test_the_token_sampler_keeps_room_for_cut_rows_alone(e3):
    logits = torch.zeros((512, 151936), dtype=torch.bfloat16, device=DEV)
    temps, side = torch.ones(512, device=DEV), torch.cuda.Stream()
    outs = e3.e3_sample(logits, temps, 1, 2)
    torch.cuda.synchronize()
    base = torch.cuda.memory_allocated()
    e3.e3_sample(logits, temps, 1, 2, out_tok=outs[0], out_logp=outs[1], out_ent=outs[2], stream=side)
    torch.cuda.synchronize()
    assert torch.cuda.memory_allocated() - base < 1 << 20


def test_many_streams_share_nothing(e3):
    streams = [torch.cuda.Stream() for _ in range(6)]
    calls = [_Calls(e3, 3 + i) for i in range(len(streams))]
    want = []
    for c, s in zip(calls, streams):
        c(s)
        want.append(c.results())
    for _ in range(30):
        for c, s in zip(calls, streams):
            c(s)
    for c, w in zip(calls, want):
        assert all(torch.equal(a, b) for a, b in zip(w, c.results()))
