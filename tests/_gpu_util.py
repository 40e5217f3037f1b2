"""Helpers for the GPU parity tests: run a synth.Workload through the C-ABI and compare with the
FP64 oracle under the three tolerances (max |err| <= 2e-2 and relative L2 <= 5e-3 on the bf16
output, |lse err| <= 1e-3)."""
import dataclasses

import numpy as np

from oracle import reference as R
from paper_2509_25224_b200 import binding

TOL_ABS = 2e-2
TOL_REL_L2 = 5e-3
TOL_LSE = 1e-3


def to_device(w):
    import torch
    dev = torch.device("cuda", 0)
    q = torch.from_numpy(w.q.view(np.int16)).to(dev).view(torch.bfloat16)
    kv = torch.from_numpy(w.kv.view(np.int16)).to(dev).view(torch.bfloat16)
    bt = torch.from_numpy(w.block_table).to(dev)
    sl = torch.from_numpy(w.seqlens).to(dev)
    return q, kv, bt, sl


def run_gpu(w, flags=None, poison=True, dev_inputs=None):
    """Returns (out float64 [B,Sq,H,512], lse float64 [B,Sq,H]) computed by the CUDA path."""
    import torch
    q, kv, bt, sl = dev_inputs if dev_inputs is not None else to_device(w)
    B, Sq, H = w.B, w.Sq, w.H
    out = torch.empty((B, Sq, H, 512), dtype=torch.bfloat16, device=q.device)
    lse = torch.empty((B, Sq, H), dtype=torch.float32, device=q.device)
    ws = torch.empty(binding.workspace_size(B, Sq, H, bt.shape[1], 0), dtype=torch.uint8, device=q.device)
    if poison:   # unwritten outputs / stale workspace must not go unnoticed
        out.view(torch.int16).fill_(0x7FC0)
        lse.fill_(float("nan"))
        ws.fill_(0xFF)
    binding.mla_decode(q, kv, bt, sl, w.scale, out, lse, ws, flags)
    binding.check_status(ws)
    torch.cuda.synchronize()
    return out.float().cpu().numpy().astype(np.float64), lse.cpu().numpy().astype(np.float64), (out, lse)


def wide_table(w, pages=4096):
    """The same workload in a block table that has room for sequences long enough for the 256-row kernel, whatever the
    lengths are (in a table as narrow as its sequences, short ones of more than 128 query rows run as blocks of 128)."""
    pad = np.full((w.B, max(0, pages - w.block_table.shape[1])), -1, np.int32)
    w.block_table = np.ascontiguousarray(np.concatenate([w.block_table, pad], axis=1))
    return w


def repeated(w, times):
    """The batch `times` times over, on the same pages: long units for every part of the schedule at the cost of one."""
    w.B *= times
    w.q = np.ascontiguousarray(np.tile(w.q, (times, 1, 1, 1)))
    w.block_table = np.ascontiguousarray(np.tile(w.block_table, (times, 1)))
    w.seqlens = np.ascontiguousarray(np.tile(w.seqlens, times))
    return w


def outside_the_cache(w, beyond):
    """(w with every second page that its sequences use outside the cache: the page `beyond` the last one, None: page -1; the same
    with those pages inside a cache that ends with a page of zeros, for the oracle)."""
    n = w.num_blocks
    bad, ref = w.block_table.copy(), w.block_table.copy()
    for b, length in enumerate(w.seqlens):
        bad[b, 0:(length + 63) // 64:2] = -1 if beyond is None else n + beyond
        ref[b, 0:(length + 63) // 64:2] = n
    zeros = np.zeros((1,) + w.kv.shape[1:], w.kv.dtype)
    return dataclasses.replace(w, block_table=bad), dataclasses.replace(w, block_table=ref, kv=np.concatenate([w.kv, zeros]))


def check_pages_outside_the_cache(w, beyond, flags=None, kernel=None):
    """A page outside the cache reads as a page of zeros, and nothing faults."""
    bad, ref = outside_the_cache(w, beyond)
    check_full(bad, flags, kernel=kernel, ref=R.decode(ref.q, ref.kv, ref.block_table, ref.seqlens, ref.scale))


def compare(out, lse, ref_out, ref_lse, what="", tol_abs=TOL_ABS):
    assert not np.isnan(out).any(), f"{what}: NaN in out"
    err = np.abs(out - ref_out)
    rel = np.linalg.norm(out - ref_out) / (np.linalg.norm(ref_out) + 1e-10)
    assert err.max() <= tol_abs, f"{what}: max|err| {err.max():.3e}"
    assert rel <= TOL_REL_L2, f"{what}: rel L2 {rel:.3e}"
    inf_ref = np.isneginf(ref_lse)
    assert np.array_equal(np.isneginf(lse), inf_ref), f"{what}: -inf pattern of lse differs"
    if (~inf_ref).any():
        le = np.abs(lse[~inf_ref] - ref_lse[~inf_ref]).max()
        assert le <= TOL_LSE, f"{what}: |lse err| {le:.3e}"
    return float(err.max()), float(rel)


def check_full(w, flags=None, what="", tol_abs=TOL_ABS, kernel=None, ref=None):
    """Every output element against the oracle (or `ref`, its results from an earlier call); `kernel`: query rows per work
    item of the kernel that has to have run."""
    out, lse, _ = run_gpu(w, flags)
    assert kernel is None or binding.last_item_rows() == kernel, (binding.last_item_rows(), kernel)
    ro, rl = ref if ref is not None else R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)
    return compare(out, lse, ro, rl, what or w.name, tol_abs)


def check_sampled(w, n_rows=192, flags=None, seed=0, what="", dev_inputs=None):
    """Full-size workloads: compare a seeded sample of (b,t,h) rows, plus finiteness everywhere."""
    out, lse, _ = run_gpu(w, flags, dev_inputs=dev_inputs)
    assert np.isfinite(out).all()
    rng = np.random.default_rng(seed)
    rows = np.stack([rng.integers(0, w.B, n_rows), rng.integers(0, w.Sq, n_rows), rng.integers(0, w.H, n_rows)], 1)
    rows = rows.astype(np.int32)
    # always include the first and last row of the first and last sequence
    rows[:4] = [[0, 0, 0], [0, w.Sq - 1, w.H - 1], [w.B - 1, 0, 0], [w.B - 1, w.Sq - 1, w.H - 1]]
    ro, rl = R.decode_rows(w.q, w.kv, w.block_table, w.seqlens, w.scale, rows)
    go = out[rows[:, 0], rows[:, 1], rows[:, 2]]
    gl = lse[rows[:, 0], rows[:, 1], rows[:, 2]]
    return compare(go, gl, ro, rl, what or w.name)
