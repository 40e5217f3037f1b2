"""CPU-side checks of the binding's argument marshalling: what it refuses, and what it hands to the library."""
import sys
import threading

import pytest
import torch

from paper_2509_25224_b200 import binding


class _FakeLibrary:
    """Stands in for the C library: records the calls instead of making them."""

    def __init__(self):
        self.calls = []

    def __getattr__(self, name):
        def call(*args):
            self.calls.append((name, args))
            return 0
        return call


@pytest.fixture
def fake(monkeypatch):
    # a process with a GPU whose current device is 0, as far as the binding can tell
    f = _FakeLibrary()
    monkeypatch.setattr(binding, "_lib", f)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: 77, raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    for name in ("_raw_stream", "_current_device"):
        if hasattr(binding, name):
            monkeypatch.setattr(binding, name, None)
    return f


def _cpu_inputs(cache_dtype):
    return (torch.zeros((1, 1, 16, 576), dtype=torch.bfloat16), torch.zeros((2, 64, 576), dtype=cache_dtype),
            torch.zeros((1, 2), dtype=torch.int32), torch.ones(1, dtype=torch.int32),
            torch.empty((1, 1, 16, 512), dtype=torch.bfloat16), torch.empty((1, 1, 16), dtype=torch.float32))


def test_host_tensors_never_reach_a_kernel(fake):
    # a host tensor's device has no index: it must not be taken for the current GPU
    q, kv, bt, sl, out, lse = _cpu_inputs(torch.bfloat16)
    with pytest.raises(ValueError):
        binding.mla_decode(q, kv, bt, sl, 0.1, out, lse, torch.empty(1 << 20, dtype=torch.uint8))
    with pytest.raises(ValueError):
        binding.mla_decode_static(q, kv, bt, sl, 0.1, out, lse)
    q, kv, bt, sl, out, lse = _cpu_inputs(torch.uint8)
    with pytest.raises(ValueError):
        binding.mla_decode_fp8(q, kv, 1.0, bt, sl, 0.1, out, lse, torch.empty(1 << 20, dtype=torch.uint8))
    assert fake.calls == []


def test_a_second_thread_may_come_in_anywhere_in_the_first_call(fake):
    # whatever the first call keeps for later ones has to be complete whenever another thread can see it: the first call is
    # held at each of its steps in turn while a second one runs
    dev = torch.device("cuda", 0)

    def held_at(step):
        binding._raw_stream = binding._current_device = None
        count, errors = [0], []

        def second():
            try:
                binding._on_device(dev, fake.anything, (), (), "second")
            except Exception as e:
                errors.append(e)

        def tracer(frame, event, arg):
            if frame.f_code is not binding._on_device.__code__:
                return None
            frame.f_trace_opcodes = True
            if event == "opcode":
                if count[0] == step:
                    t = threading.Thread(target=second)
                    t.start()
                    t.join()
                count[0] += 1
            return tracer

        before = sys.gettrace()
        sys._getframe().f_trace_opcodes = True          # Python 3.12: opcode events are on from settrace() if a frame wants them
        sys.settrace(tracer)
        try:
            binding._on_device(dev, fake.anything, (), (), "first")
        finally:
            sys.settrace(before)
        assert not errors, (step, errors)
        return count[0]

    steps = held_at(-1)
    assert steps > 20
    for step in range(steps):
        held_at(step)
