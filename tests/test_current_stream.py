"""The stream a call goes to when none is given: torch's current one, found without building a Stream object where torch allows that."""
import sys
import threading
import types

import pytest

from paper_2410_13276_b200 import binding as B


@pytest.fixture
def fake_torch(monkeypatch):
    """Stands in for torch: device 3 is current, its current stream is 77."""
    torch = types.ModuleType("torch")
    torch.cuda = types.SimpleNamespace(current_stream=lambda: types.SimpleNamespace(cuda_stream=77), current_device=lambda: 3)
    torch._C = types.SimpleNamespace(_cuda_getCurrentRawStream=lambda device: 74 + device)
    monkeypatch.setitem(sys.modules, "torch", torch)
    for name in ("_stream_handle", "_raw_stream", "_current_device"):
        if hasattr(B, name):
            monkeypatch.setattr(B, name, None)
    return torch


def test_the_current_stream_of_the_current_device(fake_torch):
    assert B._stream(None) == 77
    assert B._stream(5) == 5 and B._stream(types.SimpleNamespace(cuda_stream=6)) == 6


def test_a_torch_without_the_raw_handle(fake_torch):
    del fake_torch._C._cuda_getCurrentRawStream
    assert B._stream(None) == 77 and B._stream(None) == 77


def test_a_second_thread_at_any_point_of_the_first_call(fake_torch):
    """Another thread's call between any two instructions of a thread's first one."""
    codes = {getattr(B, n).__code__ for n in ("_current_stream", "_resolve_stream_handle") if hasattr(B, n)}
    got, seen = [], 0

    def call():
        try:
            got.append(B._stream(None))
        except Exception as e:                          # noqa: BLE001 (what it raised is what the test shows)
            got.append(repr(e))

    def at(point):
        def trace(frame, event, arg):
            nonlocal seen
            if frame.f_code not in codes:
                return None
            frame.f_trace_opcodes = True
            if event == "opcode":
                if seen == point:
                    t = threading.Thread(target=call)
                    t.start()
                    t.join()
                seen += 1
            return trace
        return trace

    before = sys.gettrace()
    sys._getframe().f_trace_opcodes = True              # (Python 3.12 traces instructions only if a frame asked for it beforehand)
    for point in range(200):
        for name in ("_stream_handle", "_raw_stream", "_current_device"):
            if hasattr(B, name):
                setattr(B, name, None)
        seen = 0
        sys.settrace(at(point))
        try:
            call()
        finally:
            sys.settrace(before)
        if seen <= point:
            break
    assert point > 10 and set(got) == {77}


@pytest.mark.gpu
def test_calls_go_to_the_stream_that_is_current():
    """A call under torch.cuda.stream is ordered behind that stream's earlier work, in threads of their own streams too."""
    import torch
    from paper_2410_13276_b200.prefill import Prefill
    streams = [torch.cuda.Stream() for _ in range(3)]
    assert B._stream(None) == torch.cuda.current_stream().cuda_stream
    for s in streams:
        with torch.cuda.stream(s):
            assert B._stream(None) == s.cuda_stream
    params = B.make_mask_params(B.SEER_TOPK_RATIO, keep_num=1, keep_den=3, flags=3)
    ref = Prefill([0, 1500], 4, 2, want_lse=False)
    scores = torch.rand(ref.scores.shape, device="cuda")
    ref.scores.copy_(scores)
    ref.mask(params)
    torch.cuda.synchronize()
    bad = []

    def work(s):
        p = Prefill([0, 1500], 4, 2, want_lse=False)
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            for _ in range(50):
                p.scores.zero_()
                p.scores.copy_(scores)                  # the mask sees this copy only from the same stream
                p.mask(params)
                n = int(p.nnz.item())
                if not (torch.equal(p.row_ptr, ref.row_ptr) and torch.equal(p.col_idx[:n], ref.col_idx[:n])):
                    bad.append(s)

    threads = [threading.Thread(target=work, args=(s,)) for s in streams]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
