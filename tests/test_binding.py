"""CPU-side checks of the binding's argument marshalling: what it refuses, and what it hands to the library."""
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
