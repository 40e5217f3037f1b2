"""GPU parity of the tensor-core decode path against the FP64 oracle, through the C-ABI, on identical
seeded inputs.  Tolerances: max |err| <= 2e-2, relative L2 <= 5e-3 (bf16 output), |lse err| <= 1e-3."""
import dataclasses

import numpy as np
import pytest

from oracle import amla_sim as S
from oracle import reference as R
from paper_2509_25224_b200 import binding, synth
from tests._gpu_util import check_full, check_sampled, repeated, run_gpu, to_device, wide_table
from tests._gpu_util import check_pages_outside_the_cache, outside_the_cache

pytestmark = pytest.mark.gpu

# every rescale variant, with the reference moved at every new maximum (tau = 0: Algorithm 2 to the
# letter) and lazily (tau = 8 octaves, the default of amla_mla_decode)
MODES = [m | binding.lazy(tau) for m in (binding.RESCALE_ALG2, binding.RESCALE_FOLD, binding.RESCALE_FMUL)
         for tau in (0, 8)] + [binding.RESCALE_ALG2 | binding.lazy(2)]


def test_config1_tiny():
    check_full(synth.config_tiny())


@pytest.mark.parametrize("n", [1, 63, 64, 65, 128, 129, 1000])
def test_single_sequence_lengths(n):
    check_full(synth.make_workload("n", 1, 1, 128, [n], seed=200 + n))


@pytest.mark.parametrize("mode", MODES)
def test_ragged_batch_all_rescale_modes(mode):
    # ragged lengths, an empty sequence, lengths shorter than Sq, Sq=2 causal rule, H=16 padding
    w = synth.make_workload("r", 6, 2, 16, [300, 0, 1, 65, 1000, 2], seed=101)
    check_full(w, mode)
    w = synth.make_workload("r", 3, 1, 128, [700, 64, 129], seed=102)
    check_full(w, mode)


@pytest.mark.parametrize("Sq,H", [(1, 16), (1, 32), (1, 64), (2, 64), (2, 128), (3, 128), (4, 128), (1, 100), (3, 50), (5, 100), (8, 128), (8, 17)])
def test_head_and_token_shapes(Sq, H):
    w = synth.make_workload("s", 3, Sq, H, [200, 77, 513], seed=300 + 10 * Sq + H)
    check_full(w)
    if Sq * H > 128:
        # (384 rows are three full blocks of 128, or two of 256 of which one is half empty: always the former)
        check_full(wide_table(w), kernel=128 if Sq * H == 384 else 256)


@pytest.mark.parametrize("lens", [[1], [64], [65], [128], [129], [191], [192], [193], [1000, 3, 0, 257, 64]])
def test_256_row_kernel_tile_tails(lens):
    # more than 128 query rows per sequence: 256-row items, 128-key tiles whose second page may be absent or partial
    w = synth.make_workload("q", len(lens), 2, 128, lens, seed=400 + sum(lens))
    check_full(w, kernel=128)
    check_full(wide_table(w), kernel=256)
    check_full(w, binding.RESCALE_ALG2 | binding.lazy(0), kernel=256)


@pytest.mark.parametrize("B,Sq,H,wide", [(31, 1, 4, False), (33, 1, 4, False), (512, 1, 2, False), (513, 1, 2, False), (65, 1, 40, False), (33, 3, 43, False), (300, 1, 33, False),
                                         (32, 2, 65, True), (65, 2, 65, True), (40, 8, 64, True), (160, 2, 65, True), (161, 2, 65, True)])
def test_schedules_worked_out_on_chip(B, Sq, H, wide):
    # items per lane of the planning warp at its edges, several row blocks per sequence, runs of empty sequences; up to and
    # beyond what is kept on chip
    lens = np.random.default_rng(B + H).integers(0, 200, B)
    lens[B // 3:B // 2] = 0
    lens[[0, -1]] = 130, 1
    w = synth.make_workload("plan", B, Sq, H, lens, seed=3000 + B + H)
    check_full(wide_table(w) if wide else w, kernel=256 if wide else 32 if Sq * H <= 32 else 128)


def test_256_row_kernel_against_128_row_blocks():
    # the same problem through both kernels (256-row items vs independent 128-row blocks): both meet the oracle
    for w in (synth.make_workload("ab", 3, 2, 128, [5000, 777, 2049], seed=431), synth.make_workload("ab4", 2, 4, 128, [3000, 130], seed=432)):
        wide_table(w)
        check_full(w, binding.DEFAULT_FLAGS, kernel=256)
        check_full(w, binding.DEFAULT_FLAGS | binding.FLAG_KERNEL_ROWS128, kernel=128)


# 400 and 500 rows: the second block of a sequence is half full, or nearly full; 1024 rows: four full blocks.  Some sequences
# are split over clusters, one begins with rows that see nothing.
@pytest.mark.parametrize("Sq,H,lens", [(4, 100, [3000, 2, 700]), (5, 100, [2000, 129, 4, 300]), (8, 128, [1500, 64, 333])])
def test_several_256_row_items_per_sequence_all_rescale_modes(Sq, H, lens):
    w = wide_table(synth.make_workload("rb", len(lens), Sq, H, lens, seed=460 + Sq))
    synth.apply_logit_offsets(w, [synth.staircase_offsets(n) if n >= 32 else np.zeros(n) for n in lens])
    ref = R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)
    for mode in MODES:
        check_full(w, mode, kernel=256, ref=ref)
    # the literal add, on inputs that leave no accumulator at zero
    w = wide_table(synth.make_workload("rbu", len(lens), Sq, H, lens, seed=465 + Sq))
    ref = R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)
    for mode in (binding.RESCALE_ALG2, binding.RESCALE_FOLD):
        check_full(w, mode | binding.lazy(0) | binding.FLAG_UNGUARDED_ADD, kernel=256, ref=ref)


def test_unguarded_add_on_zero_free_inputs():
    # the literal single integer add of Algorithm 2 line 14 (no guard for zeros): valid when no accumulator is
    # exactly zero or tiny, which N(0,1) inputs ensure
    for Sq, kernel in ((1, 128), (2, 256)):
        w = synth.make_workload("ung", 2, Sq, 128, [3000, 1500], seed=440 + Sq)
        if Sq > 1:
            wide_table(w)
        for mode in (binding.RESCALE_ALG2, binding.RESCALE_FOLD):
            check_full(w, mode | binding.lazy(0) | binding.FLAG_UNGUARDED_ADD, kernel=kernel)


def test_bounded_wait_reports_a_timeout_instead_of_hanging():
    import torch
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    binding.check_status(ws)
    binding.wait_selftest(ws, limit_ns=1_000_000)        # waits 1 ms on a barrier nothing arrives on
    with pytest.raises(binding.AmlaError) as e:
        binding.check_status(ws)
    assert e.value.code == -5
    # the context is intact and a decode on a workspace resets its status word
    check_full(synth.config_tiny())


def _check_fp8(w, kv_scale=1.0 / 64.0, flags=None, kv8=None, ref=None):
    import torch
    from tests._gpu_util import compare
    if kv8 is None:
        kv8 = synth.quantise_cache_e4m3(w, kv_scale)
    ro, rl = ref if ref is not None else R.decode_fp8(w.q, kv8, kv_scale, w.block_table, w.seqlens, w.scale)
    q, _, bt, sl = to_device(w)
    kvd = torch.from_numpy(kv8).to(q.device)
    out = torch.empty((w.B, w.Sq, w.H, 512), dtype=torch.bfloat16, device=q.device)
    lse = torch.empty((w.B, w.Sq, w.H), dtype=torch.float32, device=q.device)
    ws = torch.empty(binding.fp8_workspace_size(w.B, w.Sq, w.H, bt.shape[1], 0), dtype=torch.uint8, device=q.device)
    out.view(torch.int16).fill_(0x7FC0); lse.fill_(float("nan")); ws.fill_(0xFF)
    binding.mla_decode_fp8(q, kvd, kv_scale, bt, sl, w.scale, out, lse, ws, flags)
    binding.check_status(ws)
    torch.cuda.synchronize()
    return compare(out.float().cpu().numpy().astype(np.float64), lse.cpu().numpy().astype(np.float64), ro, rl, "fp8 " + w.name)


def test_fp8_cache_small_shapes():
    # E4M3 cache with a per-tensor scale against the FP64 oracle on the same bytes: tiny, ragged with an empty
    # sequence, two query tokens (two 128-row blocks), a scale that is not a power of two
    _check_fp8(synth.config_tiny())
    _check_fp8(synth.make_workload("f8r", 5, 1, 128, [700, 0, 64, 129, 1], seed=601))
    _check_fp8(synth.make_workload("f8q", 3, 2, 128, [1000, 65, 300], seed=602), flags=binding.RESCALE_ALG2 | binding.lazy(0))
    _check_fp8(synth.make_workload("f8s", 2, 1, 64, [500, 77], seed=603), kv_scale=0.0173)


@pytest.mark.parametrize("Sq,width,launches", [(6, 342, 3), (6, 341, 2), (8, 256, 3), (8, 255, 2), (5, 410, 2)])
def test_fp8_cache_widened_ahead_of_large_calls_of_many_rows(Sq, width, launches):
    # from six blocks of 128 rows and 8192 blocks x pages of the table on the pages are widened into a bf16 copy first
    # (a third launch); page indices outside the cache are pages of zeros on either way
    lens = [300, 0, 65, 1000]
    w = synth.make_workload("f8w", 4, Sq, 128, lens, seed=610 + Sq, spare_blocks=2 * width, max_blocks_per_seq=width)
    _check_fp8(w)
    assert binding.last_launch_count() == launches


@pytest.mark.parametrize("beyond", [0, 100000, None])
@pytest.mark.parametrize("Sq,H,kernel", [(1, 16, 32), (1, 100, 128), (2, 128, 256)])
def test_pages_outside_a_bf16_cache_are_pages_of_zeros(Sq, H, kernel, beyond):
    # the first, the last and every second page between (the 128-row kernel also asks for the next tile's pages ahead of their loads)
    w = synth.make_workload("oob", 4, Sq, H, [1500, 65, 64, 900], seed=620 + H)
    check_pages_outside_the_cache(wide_table(w) if kernel == 256 else w, beyond, kernel=kernel)


@pytest.mark.parametrize("beyond", [0, 100000, None])
@pytest.mark.parametrize("Sq,width,launches", [(1, 24, 2), (6, 342, 3)])
def test_pages_outside_an_e4m3_cache_are_pages_of_zeros(Sq, width, launches, beyond):
    # widened on their way in, and into a copy ahead of the call
    w = synth.make_workload("oob8", 4, Sq, 128, [1500, 65, 64, 900], seed=625, spare_blocks=2 * width, max_blocks_per_seq=width)
    kv8 = synth.quantise_cache_e4m3(w, 1.0 / 64.0)
    bad, ref = outside_the_cache(w, beyond)
    ref8 = np.concatenate([kv8, np.zeros((1, 64, 576), np.uint8)])
    _check_fp8(bad, kv8=kv8, ref=R.decode_fp8(ref.q, ref8, 1.0 / 64.0, ref.block_table, ref.seqlens, ref.scale))
    assert binding.last_launch_count() == launches


def test_fp8_cache_dsv3_shape_full():
    _check_fp8(synth.config_dsv3())


def test_all_sequences_empty():
    w = synth.make_workload("e", 3, 2, 128, [0, 0, 0], seed=7)
    out, lse, _ = run_gpu(w)
    assert np.all(out == 0) and np.all(np.isneginf(lse))


@pytest.mark.parametrize("H", [64, 65, 127])
@pytest.mark.parametrize("lens", [[255], [256], [257], [511, 320, 193], [1025, 31, 32, 33, 97]])
def test_128_row_kernel_tile_and_row_edges(lens, H):
    # score tiles of up to four pages whose keys the two CTAs of a cluster share page by page in halves of 32, and 64
    # query rows per CTA: lengths around a tile, a page and half a page; rows that end in the first or the second CTA
    w = synth.make_workload("edge128", len(lens), 1, H, lens, seed=450 + sum(lens) + H)
    check_full(w)
    check_full(w, binding.RESCALE_ALG2 | binding.lazy(0))


def test_many_short_sequences_more_items_than_parts():
    rng = np.random.default_rng(9)
    w = synth.make_workload("m", 200, 1, 128, rng.integers(0, 200, 200), seed=8)
    check_full(w)


def test_hundreds_of_one_page_units_per_cluster():
    # 640 sequences of 1..64 keys: every cluster runs through many one-page units back to back, so the softmax of a
    # later unit can be far ahead of the epilogue of an earlier one (the hand-off of the final scalars must hold it back)
    rng = np.random.default_rng(21)
    w = synth.make_workload("short", 640, 1, 128, rng.integers(1, 65, 640), seed=22)
    check_full(w)
    w = synth.make_workload("short2", 300, 2, 128, rng.integers(1, 130, 300), seed=23)
    check_full(w)


@pytest.mark.parametrize("B", [128, 129])
def test_items_around_the_on_chip_schedule_copy(B):
    # a full and one item more than the schedule's scan takes in four steps (the on-chip copies end at 512 items, at 160 in
    # the 256-row kernel: the tests of those are below)
    rng = np.random.default_rng(12 + B)
    w = synth.make_workload("edge", B, 1, 16, rng.integers(0, 300, B), seed=13)
    check_full(w)


@pytest.mark.parametrize("H", [16, 40])
@pytest.mark.parametrize("B", [512, 513])
def test_items_around_the_on_chip_schedule_copy_of_the_smaller_kernels(B, H):
    rng = np.random.default_rng(12 + B)
    w = synth.make_workload("edge", B, 1, H, rng.integers(0, 200, B), seed=14)
    check_full(w)


@pytest.mark.parametrize("Sq,H", [(1, 1), (1, 15), (1, 16), (1, 17), (1, 31), (2, 16), (8, 4), (3, 11)])
@pytest.mark.parametrize("lens", [[1], [63, 64, 65], [129, 127, 0, 300, 2], [5000, 700]])
def test_few_row_kernel_row_and_page_edges(lens, Sq, H):
    # up to 32 query rows (one case above): M = 64 and two score buffers up to 16 rows, M = 128 and one above; a sequence
    # begins with its Q in a slot of the page ring; masked pages; split sequences with FP32 partials
    w = synth.make_workload("few", len(lens), Sq, H, lens, seed=470 + sum(lens) + 10 * H + Sq)
    check_full(w)
    for mode in (binding.RESCALE_ALG2, binding.RESCALE_FMUL):
        check_full(w, mode | binding.lazy(0))


@pytest.mark.parametrize("Sq,H", [(1, 8), (1, 16), (2, 12), (1, 32)])
def test_few_row_kernel_rescales_within_long_units(Sq, H):
    # 160 sequences on the pages of eight: every part holds 20 to 30 pages of one or two sequences, so that O is rewritten
    # between pages.  Rising logits, a jump of 60 in the middle, falling ones; Sq = 2 masks the last page
    lens = [1500, 1400, 1279, 1344, 1600, 1217, 1000, 1537]
    w = synth.make_workload("fewr", 8, Sq, H, lens, seed=480 + H)
    plain = synth.make_workload("fewu", 8, Sq, H, lens, seed=490 + H)
    synth.apply_logit_offsets(w, [synth.staircase_offsets(n) if b % 3 == 0 else np.where(np.arange(n) < n // 2, -30.0, 30.0) if b % 3 == 1
                                  else synth.staircase_offsets(n)[::-1].copy() for b, n in enumerate(lens)])
    cases = [(w, MODES + [binding.RESCALE_ALG2]), (plain, [m | binding.lazy(0) | binding.FLAG_UNGUARDED_ADD for m in (binding.RESCALE_ALG2, binding.RESCALE_FOLD)])]
    for w, modes in cases:
        ref = [np.tile(x, (20,) + (1,) * (x.ndim - 1)) for x in R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)]
        w = repeated(w, 20)
        for mode in modes:
            check_full(w, mode, kernel=32, ref=ref)


def _unit_pages(w, parts):
    """Pages of the units (a stretch of one item in one part) that the 128-row kernel's schedule makes of a batch."""
    return {int(u[3] - u[2]) for u in binding.plan_host(w.seqlens, w.Sq, w.H, parts)}


@pytest.mark.parametrize("fp8", [False, True])
def test_128_row_kernel_rescales_over_tiles_of_every_width(fp8):
    # units of 3, 4, 5 (3 + 2), 7 (4 + 3), 8 (4 + 4) pages and more, so that O is rewritten between tiles and the keys of a CTA
    # begin in the middle of a page (tiles of three pages and of one); rising and jumping logits, tau 0 and 8
    import torch
    parts = torch.cuda.get_device_properties(0).multi_processor_count // 2
    lens = [180, 448, 512, 500, 250, 300, 700, 1250, 192, 65]
    w = synth.make_workload("pairr", len(lens), 1, 100, lens, seed=470)
    synth.apply_logit_offsets(w, [synth.staircase_offsets(n) if b % 2 else np.where(np.arange(n) < n // 2, -30.0, 30.0) for b, n in enumerate(lens)])
    kv_scale = 1.0 / 8.0
    if fp8:
        kv8 = synth.quantise_cache_e4m3(w, kv_scale)
        ref = R.decode_fp8(w.q, kv8, kv_scale, w.block_table, w.seqlens, w.scale)
    else:
        ref = R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)
    ref = [np.tile(x, (15,) + (1,) * (x.ndim - 1)) for x in ref]
    w = repeated(w, 15)
    assert {3, 4, 5, 7, 8} <= _unit_pages(w, parts)
    for mode in MODES:
        if fp8:
            _check_fp8(w, kv_scale, mode, kv8, ref)
            assert binding.last_item_rows() == 128
        else:
            check_full(w, mode, kernel=128, ref=ref)


@pytest.mark.parametrize("fp8", [False, True])
@pytest.mark.parametrize("pages", [(1, 1, 1), (4, 1, 5), (1, 9, 1, 1), (5, 6, 1, 4, 1)])
def test_128_row_kernel_units_of_one_tile_and_of_more_behind_one_another(pages, fp8):
    # the Q of a unit is asked for ahead of the epilogue of the unit two before it where one tile is all that lies between, and
    # within the unit before it else; 300 sequences, several units in every part; the last key of a page's first or second half
    import torch
    parts = torch.cuda.get_device_properties(0).multi_processor_count // 2
    lens = [64 * (pages[i % len(pages)] - 1) + (33, 64, 1, 32)[i % 4] for i in range(300)]
    w = synth.make_workload("tiles", 300, 1, 100, lens, seed=495 + len(pages))
    units = binding.plan_host(w.seqlens, 1, 100, parts)
    assert np.bincount(units[:, 0]).max() >= 4 and min(_unit_pages(w, parts)) == 1
    if fp8:
        _check_fp8(w)
    else:
        check_full(w, kernel=128)


@pytest.mark.parametrize("B,Sq,H,n", [(1, 1, 128, 400), (1, 1, 40, 4500), (1, 1, 128, 12000), (9, 1, 128, 1500), (11, 1, 128, 1500), (36, 1, 33, 700),
                                      (1, 1, 16, 20000), (36, 2, 16, 900), (75, 1, 16, 700)])
def test_merges_by_rows_and_by_quarters_of_rows(B, Sq, H, n):
    # up to 8 rows per SM a warp merges a quarter of a row, above that a row (FP32 partials: half); 2 to over 32 partials
    # per row, in one batch or several; by item and, with more items than parts, by part
    rng = np.random.default_rng(B + n)
    lens = np.maximum(1, n - rng.integers(0, n // 3, B))
    w = synth.make_workload("merge", B, Sq, H, lens, seed=600 + B + n)
    check_full(w)


@pytest.mark.parametrize("lens", [[1], [64], [65], [128], [129], [191], [192], [193], [1000, 3, 0, 257, 64], "64 short", "65 short", "160 short", "161 short", "300 short", "2100 short"])
def test_256_row_kernel_on_short_sequences_in_a_wide_table(lens):
    # short sequences of more than 128 rows are blocks of 128 rows where the table's width says that they are short, and
    # 256-row items where it does not: tile tails, and items around its on-chip and in-kernel schedules
    if isinstance(lens, str):
        lens = np.random.default_rng(31).integers(0, 130, int(lens.split()[0]))
    w = wide_table(synth.make_workload("wide", len(lens), 2, 128 if len(lens) < 100 else 65, lens, seed=500 + int(np.sum(lens))))
    check_full(w, kernel=256)
    if len(lens) < 100:
        check_full(w, binding.RESCALE_ALG2 | binding.lazy(0))


def test_few_row_kernel_reruns_are_bit_identical():
    # the lanes without a row hold leftovers of other pages: they must not have a say in when the reference moves
    w = synth.make_workload("again", 6, 1, 8, [300, 0, 1, 65, 1000, 2], seed=13)
    first = run_gpu(w)[0]
    for _ in range(10):
        assert np.array_equal(run_gpu(w)[0], first)


def test_more_items_than_the_in_kernel_schedule_handles():
    # above 2048 (sequence, row block) items the schedule prefix comes from its own kernel instead of the decode kernel
    rng = np.random.default_rng(10)
    w = synth.make_workload("big", 2100, 1, 16, rng.integers(0, 130, 2100), seed=11)
    check_full(w)


def test_more_256_row_items_than_the_in_kernel_schedule_handles():
    # the same with two query tokens and 128 heads: 2100 items of 256 rows, schedule prefix from its own kernel
    rng = np.random.default_rng(14)
    w = synth.make_workload("bigq", 2100, 2, 128, rng.integers(0, 200, 2100), seed=15)
    ref = R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)
    check_full(w, kernel=128, ref=ref)
    check_full(wide_table(w), kernel=256, ref=ref)


@pytest.mark.parametrize("mode", MODES)
def test_staircase_rescale(mode):
    check_full(synth.config_stress(B=2, N=4096), mode)


@pytest.mark.parametrize("flags", [None, binding.RESCALE_ALG2, binding.RESCALE_FOLD | binding.lazy(4)])
def test_clamp_jump_and_falling_staircase(flags):
    n = 1024
    w = synth.make_workload("j", 1, 1, 128, [n], seed=61)
    synth.apply_logit_offsets(w, [np.where(np.arange(n) < 512, -30.0, 30.0)])
    check_full(w, flags)
    w = synth.make_workload("f", 1, 1, 128, [n], seed=63)
    synth.apply_logit_offsets(w, [synth.staircase_offsets(n)[::-1].copy()])
    check_full(w, flags)


def test_exact_zero_v_columns_stay_zero():
    w = synth.config_stress(B=1, N=2048)
    w.kv[:, :, 100:110] = 0
    out, lse, _ = run_gpu(w)
    assert np.all(out[..., 100:110] == 0)
    ro, rl = R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)
    from tests._gpu_util import compare
    compare(out, lse, ro, rl, "zero columns")


def test_large_magnitude_inputs():
    # N(0, 3^2) inputs: logits spread ~ +-50, stresses the range handling of the recurrence.  The
    # softmax is then nearly one-hot and |out| reaches ~12, where half a bf16 ulp of the output alone
    # is 2^-5; the absolute tolerance is scaled with the value range (relative L2 and lse are not).
    w = synth.make_workload("g", 2, 1, 128, [2000, 700], seed=12, sigma=3.0)
    check_full(w, tol_abs=2e-2 * 4)
    w = synth.make_workload("u", 2, 1, 128, [2000, 700], seed=13, dist="uniform", sigma=5.0)
    check_full(w, tol_abs=2e-2 * 2)


def test_rerun_is_bit_identical():
    import torch
    w = synth.make_workload("d", 4, 2, 128, [3000, 1000, 64, 4097], seed=33)
    for kernel in (128, 256):
        if kernel == 256:
            wide_table(w)
        dev = to_device(w)
        _, _, (o1, l1) = run_gpu(w, dev_inputs=dev)
        _, _, (o2, l2) = run_gpu(w, dev_inputs=dev)
        assert binding.last_item_rows() == kernel
        assert torch.equal(o1.view(torch.int16), o2.view(torch.int16)) and torch.equal(l1, l2)


# The six tests from here on were written for a choice between two ways of multiplying an E4M3 cache with Q, one of which split
# Q into 8-bit numbers and is gone.  What they ask for holds for E4M3 calls in a wide table and a large cache, and in a tight one.
def _for_split_q(w, kv8):
    """(w, kv8) with a table and a cache that are large enough for the 128-row kernel to multiply K's bytes with a split Q (by the
    rule: 0.3 us a page that a part may get at most, against 1 us and 3.2 us an item)."""
    import torch
    parts = torch.cuda.get_device_properties(0).multi_processor_count // 2
    nrb = (w.Sq * w.H + 127) // 128
    pages = int((1.0 + 3.2 * w.B * nrb / parts) / 0.3 * parts / nrb) + 2
    width = max(w.block_table.shape[1], -(-pages // w.B))
    table = np.concatenate([w.block_table, np.full((w.B, width - w.block_table.shape[1]), -1, np.int32)], axis=1)
    spare = np.zeros((max(0, pages - kv8.shape[0]), 64, 576), np.uint8)
    return dataclasses.replace(w, block_table=np.ascontiguousarray(table)), np.concatenate([kv8, spare])


def _check_split_q(w, kv_scale=1.0 / 64.0, flags=None):
    kv8 = synth.quantise_cache_e4m3(w, kv_scale)
    ref = R.decode_fp8(w.q, kv8, kv_scale, w.block_table, w.seqlens, w.scale)
    big, big8 = _for_split_q(w, kv8)
    for f in flags or [None]:
        _check_fp8(big, kv_scale, f, big8, ref)
        assert binding.last_item_rows() == 128 and binding.last_launch_count() == 2


@pytest.mark.parametrize("Sq,H,lens", [(1, 128, [1]), (1, 100, [63, 64, 65, 0]), (1, 128, [128, 129, 191, 192]), (1, 128, [255, 256, 257, 320]), (2, 128, [1000, 65, 1]),
                                       (3, 43, [513, 77]), (1, 16, [700]), (5, 128, [640, 1281])])
def test_e4m3_cache_with_a_split_q(Sq, H, lens):
    # tiles of one to four pages, the middle of a page between the CTAs, several blocks of 128 rows, few rows
    _check_split_q(synth.make_workload("sq", len(lens), Sq, H, lens, seed=2600 + sum(lens)))


def test_e4m3_cache_with_a_split_q_rescales_over_tiles_of_every_width():
    lens = [180, 448, 512, 500, 250, 300, 700, 1250, 192, 65]
    w = synth.make_workload("sqr", len(lens), 1, 100, lens, seed=2610)
    synth.apply_logit_offsets(w, [synth.staircase_offsets(n) if b % 2 else np.where(np.arange(n) < n // 2, -30.0, 30.0) for b, n in enumerate(lens)])
    _check_split_q(repeated(w, 8), 1.0 / 8.0, MODES)


@pytest.mark.parametrize("pages", [(1, 1, 1), (4, 1, 5), (5, 6, 1, 4, 1)])
def test_e4m3_cache_with_a_split_q_units_behind_one_another(pages):
    # the factors on the rows' scores have four places: many units of one tile in every part
    lens = [64 * (pages[i % len(pages)] - 1) + (33, 64, 1, 32)[i % 4] for i in range(450)]
    _check_split_q(synth.make_workload("squ", 450, 1, 66, lens, seed=2620 + len(pages)))


def test_split_q_is_exact_in_the_power_of_two_of_a_row():
    # whatever power of two the rows carry, their two 8-bit parts are the same: the same bits; a row of zeros is the mean of V
    import torch
    w = synth.make_workload("sqp", 2, 1, 64, [700, 300], seed=2630)
    w.q.reshape(-1, 576)[5] = 0
    kv8 = synth.quantise_cache_e4m3(w, 1.0 / 64.0)
    ref = R.decode_fp8(w.q, kv8, 1.0 / 64.0, w.block_table, w.seqlens, w.scale)
    w, kv8 = _for_split_q(w, kv8)
    _check_fp8(w, kv8=kv8, ref=ref)
    q, _, bt, sl = to_device(w)
    kvd = torch.from_numpy(kv8).to(q.device)
    runs = [binding.mla_decode_fp8((q.float() * 2.0 ** k).to(torch.bfloat16), kvd, 1.0 / 64.0, bt, sl, w.scale * 2.0 ** -k) for k in (0, -100, 100)]
    for out, lse in runs[1:]:
        assert torch.equal(out.view(torch.int16), runs[0][0].view(torch.int16)) and torch.equal(lse, runs[0][1])


@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_an_e4m3_call_keeps_what_is_not_a_number_in_its_row(split, bad):
    # a row whose Q holds such a thing has no row sum: lse -inf, and NaN, or nothing once parts are merged; no other row notices
    import torch
    w = synth.make_workload("sqn", 2, 1, 128, [700, 300], seed=2640)
    kv8 = synth.quantise_cache_e4m3(w, 1.0 / 64.0)
    if split:
        w, kv8 = _for_split_q(w, kv8)
    q, _, bt, sl = to_device(w)
    kvd = torch.from_numpy(kv8).to(q.device)
    want, lse = binding.mla_decode_fp8(q, kvd, 1.0 / 64.0, bt, sl, w.scale)
    q[1, 0, 77, 123] = bad
    got, bad_lse = binding.mla_decode_fp8(q, kvd, 1.0 / 64.0, bt, sl, w.scale)
    row = got[1, 0, 77].clone()
    assert bad_lse[1, 0, 77] == -float("inf") and (torch.isnan(row).all() or (row == 0).all())
    got[1, 0, 77], bad_lse[1, 0, 77] = want[1, 0, 77], lse[1, 0, 77]
    assert torch.equal(got.view(torch.int16), want.view(torch.int16)) and torch.equal(bad_lse, lse)


@pytest.mark.parametrize("beyond", [0, 100000, None])
def test_pages_outside_the_cache_are_pages_of_zeros_for_a_split_q(beyond):
    w = synth.make_workload("sqo", 4, 1, 128, [1500, 65, 64, 900], seed=2650)
    w, kv8 = _for_split_q(w, synth.quantise_cache_e4m3(w, 1.0 / 64.0))
    w = dataclasses.replace(w, kv=np.zeros(kv8.shape, np.uint16))
    bad, ref = outside_the_cache(w, beyond)
    ref8 = np.concatenate([kv8, np.zeros((1, 64, 576), np.uint8)])
    _check_fp8(bad, kv8=kv8, ref=R.decode_fp8(ref.q, ref8, 1.0 / 64.0, ref.block_table, ref.seqlens, ref.scale))


def _with_room(w, kv8):
    """(w, kv8) as a serving loop has them: a table that is wider than its longest sequence, a cache of more pages than the call reads."""
    table = np.concatenate([w.block_table, np.full((w.B, max(8, 600 // w.B)), -1, np.int32)], axis=1)
    return dataclasses.replace(w, block_table=np.ascontiguousarray(table)), np.concatenate([kv8, np.zeros((6000, 64, 576), np.uint8)])


@pytest.mark.parametrize("room", [False, True])
@pytest.mark.parametrize("Sq,H,lens", [(1, 128, [1000, 65, 0, 4096]), (2, 128, [700, 2049]), (5, 77, [55, 300]), (1, 16, [20000])])
def test_an_e4m3_call_gives_the_bits_of_a_bf16_call_on_its_widened_cache(Sq, H, lens, room):
    # E4M3 values are bf16 values, so both calls have the same operands: Q in all its bits, also in rows where one element is 2^14
    # times the others and the cache has nothing in its column, so that the others are all there is
    import torch
    from tests._gpu_util import compare
    w = synth.make_workload("f8b", len(lens), Sq, H, lens, seed=2660 + Sq)
    kv8 = synth.quantise_cache_e4m3(w, 1.0 / 64.0)
    kv8[..., 570] = 0
    q = w.q.reshape(-1, 576)
    q[::2, 570] = 0x4680                                    # bf16(2^14)
    ref = R.decode_fp8(w.q, kv8, 1.0 / 64.0, w.block_table, w.seqlens, w.scale)
    if room:
        w, kv8 = _with_room(w, kv8)
    q, _, bt, sl = to_device(w)
    kvd = torch.from_numpy(kv8).to(q.device)
    flags = binding.DEFAULT_FLAGS | binding.FLAG_KERNEL_ROWS128
    out, lse = binding.mla_decode_fp8(q, kvd, 1.0, bt, sl, w.scale / 64.0, flags=flags)
    assert binding.last_item_rows() == 128
    want, want_lse = binding.mla_decode(q, kvd.view(torch.float8_e4m3fn).to(torch.bfloat16), bt, sl, w.scale / 64.0, flags=flags)
    assert binding.last_item_rows() == 128
    assert torch.equal(out.view(torch.int16), want.view(torch.int16)) and torch.equal(lse, want_lse)
    compare((out.float() / 64.0).cpu().numpy().astype(np.float64), lse.cpu().numpy().astype(np.float64), *ref, f"e4m3, wide rows, room={room}")


@pytest.mark.parametrize("fp8", [False, True])
def test_reruns_of_both_ctas_rows_are_bit_identical(fp8):
    # the MMAs of a cluster read what the warps of its odd CTA have written (P~, widened keys and values) on the word of
    # arrivals that cross to the even CTA: rising logits, so that O is rewritten too, and many units per cluster
    import torch
    w = synth.config_stress(B=20, N=1500)
    q, kv, bt, sl = to_device(w)
    if fp8:
        kv = torch.from_numpy(synth.quantise_cache_e4m3(w, 1.0 / 8.0)).to(q.device)
        ro, rl = R.decode_fp8(w.q, kv.cpu().numpy(), 1.0 / 8.0, w.block_table, w.seqlens, w.scale)
    else:
        ro, rl = R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)
    runs = []
    for _ in range(12):
        if fp8:
            runs.append(binding.mla_decode_fp8(q, kv, 1.0 / 8.0, bt, sl, w.scale))
        else:
            runs.append(binding.mla_decode(q, kv, bt, sl, w.scale))
    torch.cuda.synchronize()
    for o, l in runs[1:]:
        assert torch.equal(o.view(torch.int16), runs[0][0].view(torch.int16)) and torch.equal(l, runs[0][1])
    from tests._gpu_util import compare
    compare(runs[0][0].float().cpu().numpy().astype(np.float64), runs[0][1].cpu().numpy().astype(np.float64), ro, rl, f"rerun fp8={fp8}")


def test_matches_algorithm2_simulator_closely(capsys):
    # The CPU Algorithm-2 simulator uses the same readings; agreement should be far tighter than the oracle tolerance
    # (both round P to bf16 and accumulate in fp32).  The sequence is split over many SM groups here, and the partial
    # outputs travel in half precision (11 significant bits against the 8 of the bf16 result), so an element may land
    # on the neighbouring bf16 value: at most one bf16 unit in the last place anywhere, most elements identical.
    w = synth.config_stress(B=1, N=2048)
    out, lse, _ = run_gpu(w, binding.RESCALE_ALG2)          # tau = 0, as the simulator
    kv = synth.bf16_bits_to_f32(synth.logical_kv_rows(w, 0))
    q = synth.bf16_bits_to_f32(w.q[0, 0])
    so, sl = S.amla(q, kv, kv[:, :512], w.scale, 64)
    so = S.bf16_round(so).astype(np.float64)
    diff = np.abs(out[0, 0] - so)
    big = np.maximum(np.abs(so), np.abs(out[0, 0]))
    ulp = 2.0 ** (np.floor(np.log2(np.maximum(big, 2.0 ** -126))) - 7)      # bf16: 8 significant bits
    same = float((diff == 0).mean())
    with capsys.disabled():
        print(f"\nvs Algorithm-2 simulator: identical {same:.3f}, max diff {diff.max():.3e}, mean diff {diff.mean():.2e}")
    # one unit in the last place of the larger of the two, or (small elements of a row of large ones) the absolute
    # bound this test had with FP32 partials
    assert (diff <= np.maximum(ulp, 4e-3)).all()
    assert same >= 0.9 and diff.mean() < 1e-4
    assert np.abs(lse[0, 0] - sl).max() < 1e-4


def test_error_codes_on_device():
    import torch
    w = synth.config_tiny()
    q, kv, bt, sl = to_device(w)
    out = torch.empty((1, 1, 16, 512), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((1, 1, 16), dtype=torch.float32, device="cuda")
    small = torch.empty(1024, dtype=torch.uint8, device="cuda")
    with pytest.raises(binding.AmlaError) as e:
        binding.mla_decode(q, kv, bt, sl, w.scale, out, lse, small)
    assert e.value.code == -3
    with pytest.raises(binding.AmlaError) as e:
        binding.mla_decode(q, kv, bt, sl, w.scale, out, lse, None, flags=3)
    assert e.value.code == -1


# rows that end inside a staged block of the epilogue; 128 heads x 3 tokens are three full blocks
@pytest.mark.parametrize("entry,Sq,H,kernel", [("workspace", 1, 100, 128), ("workspace", 1, 65, 128), ("workspace", 3, 128, 128), ("workspace", 2, 75, 256),
                                               ("workspace", 2, 128, 256), ("workspace", 1, 16, 32), ("static", 1, 127, 128), ("static", 2, 100, 256),
                                               ("fp8", 1, 100, 128), ("fp8", 2, 128, 128)])
def test_outputs_that_begin_at_16_bytes(entry, Sq, H, kernel):
    # `out` need not be aligned to more than 16 bytes: a view that begins 8 elements into its buffer gets the bits that an
    # allocation of its own gets, from whole items and from merged ones, and nothing is written in front of it or behind it
    import torch
    lens = np.concatenate([np.random.default_rng(Sq * H).integers(0, 500, 90), [3000, 1, 64]])
    w = synth.make_workload("o16", len(lens), Sq, H, lens, seed=640 + Sq * H)
    if kernel == 256:
        wide_table(w, 64)
    q, kv, bt, sl = to_device(w)
    if entry == "fp8":
        kv = torch.from_numpy(synth.quantise_cache_e4m3(w, 1.0 / 64.0)).to(q.device)
    numel = w.B * Sq * H * 512
    results = []
    for first in (16, 8):
        buf = torch.full((numel + 64,), 7.0, dtype=torch.bfloat16, device=q.device)
        out = buf[first:first + numel].view(w.B, Sq, H, 512)
        lse = torch.full((w.B, Sq, H), float("nan"), dtype=torch.float32, device=q.device)
        assert out.data_ptr() % 32 == 2 * first % 32
        if entry == "fp8":
            binding.mla_decode_fp8(q, kv, 1.0 / 64.0, bt, sl, w.scale, out, lse)
        elif entry == "static":
            binding.mla_decode_static(q, kv, bt, sl, w.scale, out, lse)
        else:
            binding.mla_decode(q, kv, bt, sl, w.scale, out, lse)
        assert binding.last_item_rows() == kernel
        assert bool((buf[:first] == 7.0).all()) and bool((buf[first + numel:] == 7.0).all())
        results.append((out.clone().view(torch.int16), lse))
    assert torch.equal(results[0][0], results[1][0]) and torch.equal(results[0][1], results[1][1])


# ----------------------------------------------------------------- the five named configurations, at full size,
# every output element against the oracle (the launch configuration bench.py times)

def test_config2_dsv3_full():
    check_full(synth.config_dsv3())


def test_config3_mtp_varlen_full():
    check_full(synth.config_mtp())


def test_config4_rescale_stress_full():
    from tests._gpu_util import compare
    w = synth.config_stress()
    ro, rl = R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)
    dev = to_device(w)
    for flags in (None, binding.RESCALE_ALG2):          # the default (tau = 8) and Algorithm 2 to the letter (tau = 0)
        out, lse, _ = run_gpu(w, flags, dev_inputs=dev)
        compare(out, lse, ro, rl, f"stress flags={flags}")


def test_config5_long_context_split_full():
    from tests._gpu_util import compare
    w = synth.config_long()
    ro, rl = R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)
    dev = to_device(w)
    for flags in (None, binding.DEFAULT_FLAGS | binding.FLAG_KERNEL_ROWS128):   # 256-row kernel, and 128-row blocks
        out, lse, _ = run_gpu(w, flags, dev_inputs=dev)
        compare(out, lse, ro, rl, f"long flags={flags}")


def test_paper_grid_point_sampled():
    # one point of the paper's own benchmark grid (Section 5.2: batch 96, S_q = 2, S_k = 1024): 192 work items
    from paper_2509_25224_b200 import paper_grid
    check_sampled(paper_grid.grid_workload(2, 1024), 128)


def test_rescale_mode_accuracy_table(capsys):
    # Accuracy of the three ways to rescale O (Algorithm 2's integer add, Eq. 3's exact fold, Algorithm 1's FP32
    # multiply), each with the reference moved at every new maximum (tau = 0) and lazily (tau = 8), against the FP64
    # oracle: the paper's claim (Tables 3-4) is that the integer add costs no accuracy against the multiply.
    # Two sequences alone are cut into parts of one tile, and O is never rescaled; forty times over (on the same pages) they
    # are more items than the schedule has parts, and every unit is most of a sequence.
    cases = [(f"{name} {'x 40' if times > 1 else 'cut '}", make(), times) for times in (1, 40) for name, make in
             (("staircase B=2 N=4096", lambda: synth.config_stress(B=2, N=4096)),
              ("normal    B=2 N=8192", lambda: synth.make_workload("n", 2, 1, 128, [8192, 8192], seed=77)))]
    modes = [("alg2", binding.RESCALE_ALG2), ("fold", binding.RESCALE_FOLD), ("fmul", binding.RESCALE_FMUL)]
    lines = []
    for name, w, times in cases:
        ro, rl = (np.tile(x, (times,) + (1,) * (x.ndim - 1)) for x in R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale))
        w = repeated(w, times)
        dev = to_device(w)
        rel = {}
        for mn, mf in modes:
            for tau in (0, 8):
                out, lse, _ = run_gpu(w, mf | binding.lazy(tau), dev_inputs=dev)
                err = float(np.abs(out - ro).max())
                rel[mn, tau] = float(np.linalg.norm(out - ro) / np.linalg.norm(ro))
                le = float(np.abs(lse - rl).max())
                lines.append(f"{name} {mn:5s} tau={tau}: max|err| {err:.3e} rel_l2 {rel[mn, tau]:.3e} lse_err {le:.2e}")
                assert err <= 2e-2 and rel[mn, tau] <= 5e-3 and le <= 1e-3
        for tau in (0, 8):   # the integer add stays within 10 % of the multiply's error
            assert rel["alg2", tau] <= 1.10 * rel["fmul", tau]
    with capsys.disabled():
        print("\n" + "\n".join(lines))


def test_accuracy_grid_of_tables_3_4(capsys):
    # The paper's accuracy experiment (Section 5.1): bf16 inputs from N(0, sigma^2) and U(-a, a), 8K keys, error
    # E = |A - Golden|_F / (|Golden|_F + 1e-10), three implementations on the same inputs: Golden (here the FP64
    # oracle), Base (the CPU simulation of Algorithm 1 with bf16 P in the P V product) and AMLA (the kernel).  Ten
    # seeded samples per distribution, 16 heads of one sequence each, scale 1/sqrt(D_k) as in the paper's Eq. 1.  What
    # the paper fixes is the band its Table 3-4 values lie in (its batch, head count and block size are not stated:
    # a factor 1.12 either way around its 100-sample means) and that AMLA tracks Base.
    import math
    import os
    rows = []
    with open(os.path.join(os.path.dirname(__file__), "golden", "tables3_4_accuracy.txt")) as f:
        for line in f:
            if line.strip() and not line.startswith("#"):
                name, base, amla = line.split()
                rows.append((name, float(base), float(amla)))
    assert len(rows) == 12
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_seeds, H, N = int(os.environ.get("AMLA_ACCURACY_SEEDS", "10")), 16, 8192   # the paper averages 100 samples
    lines, checks = [], []
    for i, (name, base, amla) in enumerate(rows):
        arg = float(name[name.index(",") + 1:-1])
        dist, sigma = ("normal", math.sqrt(arg)) if name.startswith("N") else ("uniform", arg)
        e = {"base": [], "alg2": [], "fmul": [], "default": [], "alg2 whole": [], "fmul whole": []}
        for sd in range(n_seeds):
            w = synth.make_workload("acc", 1, 1, H, [N], seed=5000 + 100 * i + sd, scale=1.0 / math.sqrt(576.0), dist=dist, sigma=sigma)
            ro, rl = R.decode(w.q, w.kv, w.block_table, w.seqlens, w.scale)
            kv = synth.bf16_bits_to_f32(synth.logical_kv_rows(w, 0))
            q = synth.bf16_bits_to_f32(w.q[0, 0])
            bo, _ = S.flash_attention(q, kv, kv[:, :512], w.scale, 512, dtype=np.float32, low_precision_matmul=True)
            e["base"].append(S.rel_frobenius(S.bf16_round(bo.astype(np.float32)), ro[0, 0]))
            dev = to_device(w)
            for mn, mf in (("alg2", binding.RESCALE_ALG2 | binding.lazy(0)), ("fmul", binding.RESCALE_FMUL | binding.lazy(0)), ("default", None)):
                out, lse, _ = run_gpu(w, mf, dev_inputs=dev)
                e[mn].append(S.rel_frobenius(out, ro))
            # One sequence is cut into parts of a page each at tau = 0, and O is never rescaled; as often over as the GPU has
            # SMs, each copy is one unit of 128 pages.
            dev = to_device(repeated(w, sms))
            for mn, mf in (("alg2 whole", binding.RESCALE_ALG2 | binding.lazy(0)), ("fmul whole", binding.RESCALE_FMUL | binding.lazy(0))):
                out, lse, _ = run_gpu(w, mf, dev_inputs=dev)
                e[mn].append(S.rel_frobenius(out[sms // 2], ro[0]))
        m = {k: float(np.mean(v)) for k, v in e.items()}
        lines.append(f"{name:10s} paper base {base:.2e} amla {amla:.2e} | here ({n_seeds} seeds) base-sim {m['base']:.2e} fmul {m['fmul']:.2e} "
                     f"alg2 {m['alg2']:.2e} default(tau=8) {m['default']:.2e} whole sequences: fmul {m['fmul whole']:.2e} alg2 {m['alg2 whole']:.2e}")
        checks.append((name, base, amla, m))
    with capsys.disabled():
        print("\n" + "\n".join(lines))
    for name, base, amla, m in checks:
        assert m["alg2"] <= amla * 1.12, name
        # The lower edge only where the softmax is not one-hot: for U(-60, 60) one key takes all the weight, the
        # output is that key's bf16 row exactly, and the error against an FP64 reference vanishes.
        if name != "U(-60,60)":
            assert amla / 1.12 <= m["alg2"], name
            assert base / 1.12 <= m["base"] <= base * 1.12, name
        assert m["alg2"] <= 1.05 * m["base"] + 1e-5, name      # AMLA tracks Base (Tables 3-4)
        assert m["alg2"] <= 1.05 * m["fmul"] + 1e-5, name      # and the kernel's own FP32-multiply variant
        # The lazy reference stays with a part's first tile, so that no other key's P is 1 and exact in bf16.  Parts of one page
        # at tau = 0 ("fmul") have such a key on every page, whole sequences one in all: simulated in FP64 with only P rounded,
        # 1.86e-3 against 2.07e-3 for pages in pairs on the first one's reference.  So the bound is 1.10 times the latter.
        assert m["default"] <= 1.10 * m["fmul whole"] + 1e-5, name
        assert m["alg2 whole"] <= 1.05 * m["fmul whole"] + 1e-5, name
        assert m["alg2 whole"] <= amla * 1.12, name
