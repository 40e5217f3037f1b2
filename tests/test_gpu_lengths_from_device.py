"""Sequence lengths that a kernel directly in front of the decode call writes.

The decode kernels are launched with programmatic stream serialization and look at the lengths while they set themselves
up; what counts is what the lengths are once the kernel in front has completed.  Every call here is compared bit for bit
with the same call made on lengths that were there long before."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2509_25224_b200 import binding, synth
from tests._gpu_util import to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def late(tmp_path_factory):
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "late_lengths.cu")
    so = str(tmp_path_factory.mktemp("late") / "liblate.so")
    subprocess.check_call([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "-Xcompiler", "-fPIC", "-shared", src, "-o", so])
    f = ctypes.CDLL(so).late_lengths
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_ulonglong, ctypes.c_void_p]
    return f


# (sequences, query tokens, heads, longest, E4M3, static entry, width of the block table): the kernel for few rows, the 128-row
# kernel on either cache, 256-row items with the lengths on chip (up to 64), the prefix only (up to 160) and neither, and
# batches whose schedule is not kept on chip
CASES = [(5, 1, 16, 900, False, False, 0), (150, 1, 16, 200, False, False, 0), (6, 1, 128, 900, False, False, 0), (6, 1, 128, 900, False, True, 0),
         (40, 1, 40, 1500, False, False, 0), (5, 1, 128, 900, True, False, 0), (5, 2, 128, 900, False, False, 4096), (60, 2, 65, 400, False, False, 4096),
         (100, 2, 65, 300, False, False, 4096), (170, 2, 65, 200, False, False, 4096), (520, 1, 16, 100, False, False, 0), (520, 1, 40, 100, False, False, 0)]


@pytest.mark.parametrize("B,Sq,H,longest,fp8,static,width", CASES)
def test_lengths_written_directly_in_front_of_the_call(late, B, Sq, H, longest, fp8, static, width):
    import torch
    rng = np.random.default_rng(B + H)
    w = synth.make_workload("late", B, Sq, H, [longest] * B, seed=900 + B + H)
    if width:
        pad = np.full((B, width - w.block_table.shape[1]), -1, np.int32)
        w.block_table = np.ascontiguousarray(np.concatenate([w.block_table, pad], axis=1))
    q, kv, bt, _ = to_device(w)
    dev = q.device
    if fp8:
        kv = torch.from_numpy(synth.quantise_cache_e4m3(w, 1.0 / 64.0)).to(dev)
    size = binding.fp8_workspace_size if fp8 else binding.workspace_size
    ws = torch.empty(size(B, Sq, H, bt.shape[1], 0), dtype=torch.uint8, device=dev)
    lens = [rng.integers(0, longest + 1, B).astype(np.int32) for _ in range(3)]
    lens[0][0] = longest
    lens[1][:] = np.minimum(lens[0] + 1, longest)          # a step of a serving loop: one key more
    lens[2][0] = 0
    dlens = [torch.from_numpy(x).to(dev) for x in lens]
    garbage = torch.from_numpy(rng.integers(-2**31, 2**31 - 1, B, dtype=np.int64).astype(np.int32)).to(dev)
    seqlens = torch.empty(B, dtype=torch.int32, device=dev)

    def decode():
        out = torch.full((B, Sq, H, 512), float("nan"), dtype=torch.bfloat16, device=dev)
        lse = torch.full((B, Sq, H), float("nan"), dtype=torch.float32, device=dev)

        def go():
            if fp8:
                binding.mla_decode_fp8(q, kv, 1.0 / 64.0, bt, seqlens, w.scale, out, lse, ws)
            elif static:
                binding.mla_decode_static(q, kv, bt, seqlens, w.scale, out, lse)
            else:
                binding.mla_decode(q, kv, bt, seqlens, w.scale, out, lse, ws)
            return out, lse
        return go

    def same(a, b):
        return torch.equal(a[0].view(torch.int16), b[0].view(torch.int16)) and torch.equal(a[1], b[1])

    want = []
    for x in dlens:
        seqlens.copy_(x)
        go = decode()
        torch.cuda.synchronize()
        want.append(go())
        torch.cuda.synchronize()
    stream = torch.cuda.current_stream().cuda_stream
    # an ordinary kernel in front of every call, nothing in between: the lengths of another call, then one key more
    calls = [decode() for _ in range(24)]
    torch.cuda.synchronize()
    got = []
    for i, go in enumerate(calls):
        if i % 3 == 1:
            seqlens.add_(1).clamp_(max=longest)
        else:
            torch.add(dlens[i % 3], 0, out=seqlens)
        got.append(go())
    torch.cuda.synchronize()
    for i, g in enumerate(got):
        assert same(g, want[i % 3]), f"call {i}"
    # a kernel that lets the call start and writes the lengths 30 us later, over those of another call or over anything
    calls = [decode() for _ in range(12)]
    torch.cuda.synchronize()
    got = []
    for i, go in enumerate(calls):
        if i % 2:
            seqlens.copy_(garbage)
        assert late(dlens[i % 3].data_ptr(), seqlens.data_ptr(), B, 30000, stream) == 0
        got.append(go())
    torch.cuda.synchronize()
    for i, g in enumerate(got):
        assert same(g, want[i % 3]), f"late call {i}"
    if static:
        binding.static_check_status()
    else:
        binding.check_status(ws)


@pytest.mark.parametrize("B,Sq,H,longest,fp8,width", [(40, 3, 128, 600, True, 0), (25, 3, 128, 900, False, 4096), (70, 3, 43, 500, True, 0), (60, 5, 128, 400, False, 4096)])
def test_lengths_written_while_a_call_of_several_row_blocks_starts(late, B, Sq, H, longest, fp8, width):
    # the items of a sequence load its length one by one: the write falls before, among and behind these loads
    import torch
    rng = np.random.default_rng(B)
    w = synth.make_workload("blocks", B, Sq, H, [longest] * B, seed=950 + B)
    if width:
        pad = np.full((B, width - w.block_table.shape[1]), -1, np.int32)
        w.block_table = np.ascontiguousarray(np.concatenate([w.block_table, pad], axis=1))
    q, kv, bt, _ = to_device(w)
    dev = q.device
    if fp8:
        kv = torch.from_numpy(synth.quantise_cache_e4m3(w, 1.0 / 64.0)).to(dev)
    size = binding.fp8_workspace_size if fp8 else binding.workspace_size
    ws = torch.empty(size(B, Sq, H, bt.shape[1], 0), dtype=torch.uint8, device=dev)
    dlens = [torch.from_numpy(rng.integers(0, longest + 1, B).astype(np.int32)).to(dev) for _ in range(2)]
    seqlens = torch.empty(B, dtype=torch.int32, device=dev)
    out = torch.empty((B, Sq, H, 512), dtype=torch.bfloat16, device=dev)
    lse = torch.empty((B, Sq, H), dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream().cuda_stream

    def call_behind(write):
        out.fill_(float("nan"))
        lse.fill_(float("nan"))
        write()
        if fp8:
            binding.mla_decode_fp8(q, kv, 1.0 / 64.0, bt, seqlens, w.scale, out, lse, ws)
        else:
            binding.mla_decode(q, kv, bt, seqlens, w.scale, out, lse, ws)
        torch.cuda.synchronize()
        return out.view(torch.int16).clone(), lse.clone()

    want = [call_behind(lambda x=x: seqlens.copy_(x)) for x in dlens]
    for i, delay in enumerate(range(0, 16000, 400)):
        seqlens.copy_(dlens[1 - i % 2])
        code = []
        got = call_behind(lambda: code.append(late(dlens[i % 2].data_ptr(), seqlens.data_ptr(), B, delay, stream)))
        assert code == [0]
        assert torch.equal(got[0], want[i % 2][0]) and torch.equal(got[1], want[i % 2][1]), (i, delay)
    binding.check_status(ws)
