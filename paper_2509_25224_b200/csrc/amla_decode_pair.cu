// Tensor-core MLA decode kernel for sequences of up to 128 query rows, sm_100a.
//
// A cluster of two CTAs works on one 128-row block of query rows and a range of 64-key cache pages.  Both CTAs do the
// same work on 64 rows each; every matrix product is an MMA over the pair (tcgen05.mma.cta_group::2, M = 128, N up to
// 256), so each CTA supplies its own 64 rows of A and HALF of the B operand:
//
//   S = Q K^T     A = Q (64 rows x 576, shared memory), B = K: CTA j loads the first or second half of a tile's keys
//   O += P~ V     A = P~ (64 rows x 64 keys per page, shared memory), B = V: CTA j loads columns 256 j .. 256 j + 255
//
// With M = 128 over two CTAs the accumulators use all 128 tensor-memory lanes of either CTA: lanes 0-63 hold the CTA's
// 64 rows for the first half of the N columns, lanes 64-127 the same rows for the second half.  S of four pages
// (256 keys) takes 128 columns, O (512 columns of V) takes 256, so S is double buffered and Q need not go into tensor
// memory: it is an operand as soon as TMA has delivered it.
//
// Warps 0-7 run Algorithm 2's recurrence (lines 5-12; four threads share a query row: lane half = half of a tile's keys,
// warp group = even / odd pages), write P~ = bf16(P * S16) into the P buffer of their own CTA, apply the integer N to
// the bit patterns of O when the row's reference moved (lines 13-16; Lemma 3.1) and run the epilogue (line 20).  They
// never hand data to the other CTA.  Warps 8, 10 and 11 load (TMA), warp 9 of the even CTA issues the MMAs for both.
// Order on the tensor pipe: QK^T(i + 1) before P~V(i) (the paper's [C1, C2, V1] order, Section 4.1), whether or not the two
// tiles belong to one unit: the next unit's Q is asked for as soon as the scores of a unit's last tile are there, and its first
// scores are made while those are worked on.  (Each unit a chain by itself: 1 x 2531 keys 13.09 -> 12.78 us, 29 x 238-661
// 18.95 -> 18.69, 32 x 4096 55.75 -> 55.21, E4M3 61.8 -> 60.5; outputs the same bits.)
//
// Why this split.  The kernel before it gave one CTA of the pair Q K^T and the other P~ V (M = 128 on one SM each): P~
// crossed to the other SM by remote stores, Q went through shared memory into tensor memory and the score CTA had to be
// drained before the next unit's Q could follow.  Here nothing but MMA operands crosses, Q is an operand as it lands, and
// the tile is 256 keys.  Calls with it, from that kernel to this one as it stands (sustained): 192 sequences of 1-512 keys
// 62.8 -> 38.1 us; one of 2531 33.8 -> 12.3; 16 x 16384 with rising logits 106.0 -> 93.7; 96 x 2048 88.7 -> 78.4; 32 x 4096
// 59.1 -> 53.2; E4M3 32 x 4096 100.4 -> 60.4.  (The last of each pair from one GPU; others are up to 3 % faster.)
// What bounds it (trace): a tile of 256 keys takes 7100 clk in long units, 7600 on average over the eight of a 32 x 4096 call,
// against 4350 of MMAs, 5600 of shared memory at 128 bytes a clk (MMA operands 408 KB, TMA 278, P~ 32) and 5900-6600 of HBM.  The
// issuer finds every slot full that it comes to, and takes 350 clk for a slot of K and 390 for one of V, 17 of them a tile: the
// operands of four MMAs and the 16 KB that TMA writes meanwhile are 320 clk of shared memory.  E4M3: a tile is 17 slots of ~575 clk,
// 996 KB through shared memory (7800 clk), and two of the four schedulers convert 17 x 352 clk beside the softmax.  Long calls run
// at the power limit, at 1.4-1.75 GHz: 32 x 4096 takes 48.5 us cool.
//
// All waits are bounded; on expiry the kernel records kStatusTimeout and unwinds.
#include "amla_common.cuh"
#include "amla_host.cuh"
#include "amla_sm100.cuh"
#include "amla_epilogue.cuh"
#include "amla_units.cuh"

namespace amla {

using namespace sm100;

namespace {

constexpr int kSoftmaxWarps = 8;
// bf16 cache: warps 8, 10 and 11 load.  E4M3 cache: warp 8 loads (more warps would leave too few registers), warps 10-15
// widen, three pairs taking turns.
constexpr int kWidenGroups = 3, kWidenWarps = 2;
constexpr int kWideners = kWidenGroups * kWidenWarps;
constexpr int kLoaders = 3;
template <bool kFp8> constexpr int kThreads = 32 * (kFp8 ? kSoftmaxWarps + 2 + kWideners : kSoftmaxWarps + 1 + kLoaders);
constexpr int kTilePages = 4;                           // pages of a score tile: N = 256, the widest MMA
constexpr int kCtaRows = kRowBlock / 2;                 // query rows per CTA
constexpr int kQBlocks = kDqk / 64;                     // 64-column blocks of Q and K
constexpr uint32_t kQBlockBytes = kCtaRows * 128;       // [64 rows][128 B], 128-byte swizzle
constexpr uint32_t kQBytes = kQBlocks * kQBlockBytes;
constexpr uint32_t kPPageBytes = kCtaRows * 128;        // P~ of one page: [64 rows][64 keys]
constexpr uint32_t kKBoxBytes = 32 * 128;               // half a page (32 keys) x one 64-column block
constexpr uint32_t kSlotBytes = 128 * 128;              // K: half of 4 pages' keys x 64 columns; V: 64 keys x 128 columns
constexpr uint32_t kVBlockBytes = 64 * 128;             // 64 keys x 64 columns
// The ring of operand slots, and for an E4M3 cache a ring of raw slots in front of it, one for every two operand slots.
// A rule that every user of a ring keeps: a thread waits only for slots that it fills or empties itself, and having waited
// for number w (counted over the whole run; slots are released in order) next for one of w + 1 ... w + R, R being the number
// of slots.  The barriers tell two successive phases apart, no more: a thread that asks for a phase further on is let
// through by an older one, and one that comes to ask after the next phase has passed as well is held for good.  (So the
// three loaders take every third number on a ring of seven slots, and the three pairs that widen step by three through four operand
// slots, and so by one or two through three raw slots.  Raw slots are filled in any order, since V comes from L2 and K from HBM, so
// a pair waits for its operand slot first: that it is free says which raw slots had been full.)
template <bool kFp8> constexpr int kSlots = kFp8 ? 4 : 7;
constexpr int kRawSlots = 3;
constexpr uint32_t kRawBytes = kSlotBytes;              // the bytes of two operand slots

constexpr uint32_t kOffQ = 0;
constexpr uint32_t kOffP = kOffQ + kQBytes;
constexpr uint32_t kOffRing = kOffP + kTilePages * kPPageBytes;
constexpr uint32_t kOffRaw = kOffRing + kSlots<true> * kSlotBytes;
constexpr uint32_t kOffXchg = kOffRing + 7 * kSlotBytes;           // float [2][4 threads of a row][64 rows]
static_assert(kOffRaw + kRawSlots * kRawBytes <= kOffXchg && kSlots<false> <= 7, "the rings share one area");
constexpr uint32_t kOffBars = kOffXchg + 2 * 4 * kCtaRows * 4;
constexpr uint32_t kBarBytes = 384;
// a copy of the schedule prefix and of the sequence lengths for batches of up to kSmemPlanItems items, so that the
// roles' schedule look-ups (a dozen dependent loads per unit) stay on chip
constexpr int kSmemPlanItems = 512;
constexpr uint32_t kOffPlan = kOffBars + kBarBytes;
constexpr uint32_t kOffSeqlens = kOffPlan + ((kSmemPlanItems + 1) * 4 + 15) / 16 * 16;
constexpr uint32_t kOffFirst = kOffSeqlens + kSmemPlanItems * 4;
constexpr uint32_t kSmemBytes = kOffFirst + sizeof(FirstUnit);
static_assert(kSmemBytes <= 232448, "exceeds the shared memory a block can opt in to");
static_assert(kOffP % 1024 == 0 && kOffRing % 1024 == 0, "swizzled tiles need 1024-byte alignment");

// tensor-memory columns
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kOCol = 0;            // 256 columns
constexpr uint32_t kSCol = 256;          // 2 x 128 columns

// Barriers.  (L): the copy in the even CTA is the one that counts; both CTAs arrive there.  The others exist in both
// CTAs and complete by multicast commits of the even CTA's MMA warp, except X_XCHG and the raw ring's, which are local.
enum { X_FULL = 0 /*L*/, X_EMPTY = X_FULL + 7, X_QFULL = X_EMPTY + 7 /*L*/, X_SFULL, X_SEMPTY = X_SFULL + 2 /*L*/,
       X_PREADY = X_SEMPTY + 2 /*L*/, X_PVDONE, X_XCHG, X_RAWFULL = X_XCHG + 2, X_RAWEMPTY = X_RAWFULL + kRawSlots,
       X_FULLODD = X_RAWEMPTY + kRawSlots /* odd CTA, E4M3: its half of FULL, passed on */, X_NUM = X_FULLODD + kSlots<true> };
static_assert(X_NUM * 8 + 8 <= kBarBytes, "barrier area too small");

__device__ __forceinline__ void report_timeout(int* status) { atomicExch(status, kStatusTimeout); }

// Wait whose verdict is the same in every lane of the warp, so that the warp-collective tensor-memory instructions
// that follow are never executed by a part of it.
template <bool kClusterAcquire = false>
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait<kClusterAcquire>(bar, parity));
}

using Tiles = TileIter<kTilePages>;

// The page numbers of a tile.
static_assert(kTilePages == 4, "a tile's page numbers");
struct Pages { int a, b, c, d; };
__device__ __forceinline__ Pages load_pages(const DecodeParams& prm, const Tiles& tile) {
  Pages pg = {};
  if (tile.valid) {
    const int32_t* bt = prm.block_table + static_cast<size_t>(tile.u.b) * prm.max_blocks_per_seq + tile.t;
    pg.a = ldg_here(bt);
    if (tile.np > 1) pg.b = ldg_here(bt + 1);
    if (tile.np > 2) pg.c = ldg_here(bt + 2);
    if (tile.np > 3) pg.d = ldg_here(bt + 3);
  }
  return pg;
}

// This CTA's 64 rows of a unit's Q, by one thread of either CTA.  The bytes of both are counted in the even one.
__device__ __forceinline__ int q_row_of(const DecodeParams& prm, const Unit& u, int rank) { return u.b * prm.R + u.r0 + rank * kCtaRows; }
__device__ __forceinline__ void request_q(const CUtensorMap& q_map, uint32_t smem_base, uint32_t bars, uint32_t lead_bars, bool leader, int qrow) {
  if (leader) mbar_arrive_expect_tx(bars + 8u * X_QFULL, 2 * kQBytes);
  const uint64_t last_use = l2_policy_evict_first();
#pragma unroll 1
  for (int c = 0; c < kQBlocks; c += 3)
    tma_load_3d_pair_hint(smem_base + kOffQ + c * kQBlockBytes, &q_map, 0, qrow, c, lead_bars + 8u * X_QFULL, last_use);
}

}  // namespace

template <int kMode, bool kGuard, bool kFp8>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads<kFp8>, 1)
decode_pair_kernel(const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap khalf_map, const __grid_constant__ CUtensorMap v_map, const __grid_constant__ CUtensorMap q_map,
                   const DecodeParams prm) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t smem_base = smem_u32(smem_raw);
  const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const bool leader = rank == 0;
  const int part = blockIdx.x >> 1;
  if (tid == 0 && leader) AMLA_STAMP(prm, part, 20, 0);
  if (smem_base & 1023u) {   // the swizzled tiles assume a 1024-byte aligned window; identical in both CTAs
    if (tid == 0) report_timeout(prm.status);
    return;
  }
  const uint32_t bars = smem_base + kOffBars;
  auto bar = [&](int i) { return bars + 8u * i; };
  const uint32_t tmem_slot = bars + kBarBytes - 8;
  const uint32_t lead_bars = map_to_cta(bars, 0);

  // Set-up.  The schedule of a batch of up to kSmemPlanItems items is worked out from the sequence lengths as they are found
  // (held against the final ones after the wait below): all threads bring them, or warp 8 where they are few, and warp 8 adds up.
  // Beside that warp 9 allocates tensor memory and one thread of warp 10 initialises the barriers.
  const bool plan_here = prm.fused_plan && prm.n_items <= kSmemPlanItems;
  int* plan_smem = reinterpret_cast<int*>(smem_raw + kOffPlan);
  int* lens_smem = reinterpret_cast<int*>(smem_raw + kOffSeqlens);
  FirstUnit* first_smem = reinterpret_cast<FirstUnit*>(smem_raw + kOffFirst);
  const bool by_warp = prm.n_items <= kWarpPlanItems;
  if (plan_here && (!by_warp || wid == 8)) plan_lengths(prm, plan_smem, lens_smem, by_warp ? lane : tid, by_warp ? 32 : kThreads<kFp8>);
  if (tid == 32 * 10) {
    for (int i = 0; i < kSlots<kFp8>; ++i) {
      mbar_init(bar(X_FULL + i), kFp8 ? kWidenWarps + 1 : 1);          // E4M3: the warps that fill the slot, and word from the odd CTA
      mbar_init(bar(X_EMPTY + i), 1);
      if (kFp8) mbar_init(bar(X_FULLODD + i), kWidenWarps);
    }
    if (kFp8) {
      for (int i = 0; i < kRawSlots; ++i) { mbar_init(bar(X_RAWFULL + i), 1); mbar_init(bar(X_RAWEMPTY + i), 2 * kWidenWarps); }
    }
    mbar_init(bar(X_QFULL), 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(X_SFULL + i), 1);
      mbar_init(bar(X_SEMPTY + i), 2 * kSoftmaxWarps);
      mbar_init(bar(X_XCHG + i), kSoftmaxWarps / 2);
    }
    mbar_init(bar(X_PREADY), 2 * kSoftmaxWarps);
    mbar_init(bar(X_PVDONE), 1);
    fence_mbar_init();
    prefetch_tensormap(&k_map);
    prefetch_tensormap(&khalf_map);
    prefetch_tensormap(&v_map);
    prefetch_tensormap(&q_map);
  }
  if (wid == 9) { tmem_alloc_pair(tmem_slot, kTmemCols); tmem_relinquish_pair(); }
  if (tid == 0 && leader) AMLA_STAMP(prm, part, 20, 6);
  if (plan_here) {
    if (by_warp) __syncwarp(); else __syncthreads();
    if (wid == 8) plan_units(prm, plan_smem, lens_smem, first_smem, part, lane);
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_arrive_relaxed();        // the peer's barriers are initialised before anyone signals them (waited for below)
  tc_fence_after_sync();
  const uint32_t tbase = ld_shared_b32(tmem_slot);
  if (tid == 0 && leader) AMLA_STAMP(prm, part, 20, 3);

  const int* prefix = plan_here ? plan_smem : prm.prefix;
  const int* seqlens = plan_here ? lens_smem : prm.seqlens;
  if (!plan_here) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    if (prm.fused_plan) {      // (kSmemPlanItems, kFusedPlanMaxItems] items: every CTA writes the same prefix to the workspace
      if (wid == 0) {
        plan_in_workspace(prm, lane);
        if (tid == 0 && blockIdx.x == 0) *prm.status = kStatusOk;
        __threadfence_block();
      }
      __syncthreads();
    }
  }
  bool ok = true;
  Tiles tile(UnitIter(prm, prefix, seqlens, part), plan_here ? first_smem : nullptr);
  if (tid == 0 && leader) AMLA_STAMP(prm, part, 20, 5);
  cluster_wait();
  Pages first_pages = {};                                    // the loaders' first tile: on their way while the lengths are
  if (!plan_here) {
    if (wid >= kSoftmaxWarps) first_pages = load_pages(prm, tile);
  } else {
    // Launched with programmatic stream serialization: everything above ran while the kernel before this one on the stream
    // was still going; its results (the previous call's reads of the workspace among them) are complete after this wait.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    if (wid >= kSoftmaxWarps) first_pages = load_pages(prm, tile);     // (the guess's place in the table is inside the table)
    if (plan_is_stale(prm, plan_smem, lens_smem, first_smem, tid, kThreads<kFp8>)) {     // (both CTAs see the same lengths)
      plan_lengths(prm, plan_smem, lens_smem, tid, kThreads<kFp8>);
      __syncthreads();
      if (wid == 8) plan_units(prm, plan_smem, lens_smem, first_smem, part, lane);
      __syncthreads();
      tile.start(first_smem);
      if (wid >= kSoftmaxWarps) first_pages = load_pages(prm, tile);
    }
    if (blockIdx.x == 0 && wid == 0 && lane == 0) *prm.status = kStatusOk;
  }
  if (tid == 0 && leader) AMLA_STAMP(prm, part, 20, 4);

  if (wid < kSoftmaxWarps) {
    // ======================================================== softmax, correction, epilogue
    const int quarter = wid & 3, grp = wid >> 2;
    const int khalf = quarter >> 1;                      // S: key half of every page; O: which 256 columns
    const int r = (quarter & 1) * 32 + lane;             // query row within this CTA's 64
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    const bool scale_nonneg = prm.scale_log2 >= 0.f;
    const uint32_t xbar = bar(X_XCHG + (quarter & 1));
    const uint32_t prow_smem = smem_base + kOffP + r * 128;
    const uint32_t o_addr = tbase + lane_base + kOCol + 128 * grp;     // this thread's 128 of the row's 512 columns
    uint32_t gs = 0, xc = 0;                             // score tiles and exchanges so far
    // Warp 7 asks for the next unit's Q as soon as the scores of a unit's last tile are there: the MMAs have then read Q.
    // It looks the unit up well before that.  For a unit of one tile that is ahead of the epilogue of the unit before, as it has
    // to be: that unit's last P~V is followed by the Q K^T that the Q is for.  (Behind that epilogue: 60 x 55 keys, five tokens
    // 43.8 -> 48.2 us, 192 x 1-512 42.2 -> 43.8.)
    constexpr int kAsksForQ = 7;
    uint32_t q_asked = 0;                                // units whose Q this warp has asked for
    int q_next = -1;                                     // first row of the next unit's Q, -1: there is none, or it has been asked for
    auto look_ahead = [&]() {
      UnitIter ahead = tile.units;                       // stands behind the unit that tile is in
      Unit n;
      q_next = ahead.next(n) ? q_row_of(prm, n, rank) : -1;
    };
    auto ask_for_q = [&]() {                             // the scores of the last tile before that unit are there
      if (lane == 0) request_q(q_map, smem_base, bars, lead_bars, leader, q_next);
      __syncwarp();                                      // what follows is the whole warp's
      ++q_asked;
      q_next = -1;
    };
    if (wid == kAsksForQ && tile.valid) look_ahead();
    // tells the row's other three threads `mine`; v[0..3] = what the four told
    auto exchange = [&](float mine, float (&v)[4]) {
      const uint32_t buf = smem_base + kOffXchg + (xc & 1) * (4 * kCtaRows * 4) + r * 4;
      st_shared_b32(buf + (2 * khalf + grp) * (kCtaRows * 4), __float_as_uint(mine));
      __syncwarp();
      if (lane == 0) mbar_arrive(xbar);
      ok = warp_wait(xbar, xc & 1);
      ++xc;
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(ld_shared_b32(buf + i * (kCtaRows * 4)));
    };
    // the same without a word: the row group's four warps have all come here
    auto group_sync = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(xbar);
      ok = warp_wait(xbar, xc & 1);
      ++xc;
    };
    // 32 keys of P~: half (chunk & 1) of page chunk / 2 of the P buffer, in pieces of 8
    auto store_p_piece = [&](int chunk, int c, const uint32_t (&pk)[16]) {
      st_shared_v4(prow_smem + (chunk >> 1) * kPPageBytes + (((4 * (chunk & 1) + c) ^ (r & 7)) << 4), pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
    };

    if (tid == 0 && leader) merge_begin(prm, part);
    write_empty_items(prm, prefix, part, prm.P, rank * kCtaRows, kCtaRows, tid, 32 * kSoftmaxWarps);
    // A tile's softmax is done while the P~V of the tile before it still runs, and so is, at the end of a unit, that of the next
    // unit's first tile ahead of the unit's own epilogue: P~ then waits in the columns that its scores had, and is copied into the
    // P buffer when that P~V has read it.  What is left between two P~V is the epilogue or the rescale, and the copy.  Against
    // exponentials behind that P~V and units whose softmax began behind the epilogue of the one before: 192 x 1-512 keys 38.8 ->
    // 37.3 us, 60 x 55 with five tokens 38.3 -> 36.8, 150 x 1-128 with two 40.1 -> 38.1, 16 x 16384 86.3 -> 84.6, 96 x 2048 73.5 ->
    // 72.5, 32 x 4096 50.4 -> 49.8; E4M3 32 x 4096 58.4, so 58.4.  (Only at the ends of units: 38.0, 87.6, 73.3, 50.3.)
    RowState st;
    row_state_init(st);
    int visible = 0, first_masked = 0;
    int e_row = -1, e_b = 0, e_slot = 0;                 // the unit whose epilogue is still to be done: this thread's row (-1: none), ...
    float e_inv = 0.f, e_lse = 0.f;
    while (tile.valid || e_row >= 0) {
      const uint32_t sb = gs & 1;
      const int t = tile.t, np = tile.np;
      // A lane half holds 32 np neighbouring keys of a tile; this group takes its 32-key chunks grp and grp + 2.
      const uint32_t scol = tbase + lane_base + kSCol + 128 * sb + 32 * grp;
      const int chunk0 = np * khalf + grp;                                  // of the tile's 2 np
      // P~ goes straight into the P buffer, 8 keys at a time as they are ready; into tensor memory 32 at a time, with an E4M3 cache,
      // where registers are few, 8.  (32 / 8: E4M3, 1 x 130 keys 10.73 / 10.62 us, 1 x 256 10.99 / 10.90, 8 x 1000 with 16 heads 14.38 /
      // 14.23; bf16, 8 at a time: 1 x 256 with 16 heads 7.87 / 7.95, 192 x 1-512 32.6 / 32.8.)
      bool direct = false;
      uint32_t nword = 0;
      bool moved = false;
      if (tile.valid) {
        if (tile.first) {
          const Unit& u = tile.u;
          row_state_init(st);
          const int tok = (u.r0 + rank * kCtaRows + r) / prm.H;
          visible = min(u.n_b, u.n_b - prm.Sq + tok + 1);          // keys 0..visible-1 are seen by this row
          first_masked = max(u.n_b - prm.Sq + 1, 0) / kPage;       // pages from here on may hold hidden keys
        }
        ok = warp_wait(bar(X_SFULL + sb), (gs >> 1) & 1);
        if (!ok) break;
        tc_fence_after_sync();
        if (tid == 0 && leader) AMLA_STAMP(prm, part, 8, gs);
        if (wid == kAsksForQ && tile.last() && q_next >= 0) ask_for_q();
        // The scores are read from tensor memory twice, a chunk at a time: for the maximum, and for the exponentials.  (Held in
        // registers in between they cost 64 more of them and twice the code.)
        const int nvis0 = visible - t * kPage - 32 * chunk0;                // keys of the first chunk that the row sees (may be <= 0)
        const bool plain = t + np <= first_masked && scale_nonneg;          // every key of the tile is visible
        // lines 5-6: running max (the scale is folded into the FMA below)
        float ext = -INFINITY;
#pragma unroll 1
        for (int h = 0; grp + 2 * h < np && h < 2; ++h) {
          uint32_t v[32];
          tmem_ld_32x32b_x32(scol + 64 * h, v);
          tmem_wait_ld();
          float a = -INFINITY, b = a;
          if (plain) {
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              a = fmax3(a, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
              b = fmax3(b, __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
            }
            a = fmaxf(a, b) * prm.scale_log2;
          } else {
            const int nvis = nvis0 - 64 * h;
#pragma unroll
            for (int i = 0; i < 32; ++i) a = fmaxf(a, i < nvis ? __uint_as_float(v[i]) * prm.scale_log2 : -INFINITY);
          }
          ext = fmaxf(ext, a);
        }
        float m4[4];
        exchange(ext, m4);
        if (!ok) break;
        if (tid == 0 && leader) AMLA_STAMP(prm, part, 9, gs);
        const float tmax = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
        // Lazy reference: a row must move when its maximum exceeds the reference by more than tau.  The four warps of these
        // 32 rows pay for a rescale as soon as one row moves, so when one must, every row of the warp whose maximum rose
        // moves with it (moving early is always allowed: tau = 0 moves at every rise); the rows then tend to stay in step and
        // O is rescaled on far fewer tiles.  The four warps see the same maxima and agree.
        const bool must = tmax > st.m2 + prm.tau;
        const RowStep sp = row_step<kMode>(st, tmax, __any_sync(0xffffffffu, must) ? 0.f : prm.tau);
        nword = (kMode == 2) ? __float_as_uint(sp.l_up) : static_cast<uint32_t>(sp.n_bits);
        moved = !tile.first && __any_sync(0xffffffffu, (kMode == 2) ? (sp.l_up != 1.f) : (sp.n_bits != 0));
        direct = gs == 0 || (e_row < 0 && !moved && __all_sync(0xffffffffu, mbar_probe(bar(X_PVDONE), (gs - 1) & 1)));
        // Line 10's factor S16 goes into the exponential's argument (the remark after Algorithm 2).  The row sum of line 6 is
        // the sum of the same FP32 values, taken before the bf16 cast and divided by S16 once per tile.
        const float nsub = log2f_approx(sp.p_scale) - sp.m2_sub;
        const float sc = plain ? prm.scale_log2 : 1.f;
        const uint64_t sc2 = pack_f32x2(sc, sc), ns2 = pack_f32x2(nsub, nsub);
        uint64_t rsa = pack_f32x2(0.f, 0.f), rsb = rsa;
#pragma unroll 1
        for (int h = 0; grp + 2 * h < np && h < 2; ++h) {
          uint32_t v[32];
          tmem_ld_32x32b_x32(scol + 64 * h, v);
          tmem_wait_ld();
          if (!plain) {
            const int nvis = nvis0 - 64 * h;        // scaled here; hidden keys become 2^-inf = 0
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = i < nvis ? __float_as_uint(__uint_as_float(v[i]) * prm.scale_log2) : 0xff800000u;
          }
          uint32_t pk[16];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
#pragma unroll
            for (int i = 4 * c; i < 4 * c + 4; ++i) {
              float x0, x1;
              unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])), sc2, ns2), x0, x1);
              const float q0 = ex2_approx(x0), q1 = ex2_approx(x1);
              const uint64_t pp = pack_f32x2(q0, q1);
              if (i & 1) rsb = add_f32x2(rsb, pp); else rsa = add_f32x2(rsa, pp);
              pk[i] = pack_bf16x2(q0, q1);
            }
            if (direct) store_p_piece(chunk0 + 2 * h, c, pk);
            else if (kFp8) tmem_st_32x32b_x4(scol + 64 * h + 4 * c, pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
          }
          if (!kFp8 && !direct) tmem_st_32x32b_x16(scol + 64 * h, pk);
        }
        float s0, s1;
        unpack_f32x2(add_f32x2(rsa, rsb), s0, s1);
        st.l = st.l * sp.l_up + __fdividef(s0 + s1, sp.p_scale);   // this thread's share of the row sum
      }
      if (!direct) {
        // the P~V of the tile before: it has read the P buffer, and O holds its sum
        tmem_wait_st();
        ok = warp_wait(bar(X_PVDONE), (gs - 1) & 1);
        if (!ok) break;
        tc_fence_after_sync();
        if (e_row >= 0) {
          // ---- epilogue (line 20): out = O / (l * S16), lse = m + ln l.  Thread = row; the four threads of a row take 128
          // of its 512 columns each.
          if (tid == 0 && leader) AMLA_STAMP(prm, part, 13, gs - 1);
          const bool valid = e_row < prm.R;
          const int col0 = 256 * khalf + 128 * grp;
          const int prow0 = (e_slot < 0 ? 0 : e_slot) * kRowBlock + rank * kCtaRows;   // this CTA's first row of the partial arrays
          // The warp's 32 rows x 64 columns at a time pass through the rows of the P buffer that belong to this row group (P~V has
          // read them; the group writes them again only when all of its warps are done here), so that a store covers 128 bytes of
          // four rows: whole lines leave the SM at about twice the rate of 32-byte pieces of 32 rows.  A lane stores 16 bytes, which
          // is what `out` is aligned to (32 bytes of eight rows are no faster: 192 x 1-512 keys 43.98 us, so 44.00; 60 x 55, five
          // tokens 48.2, 48.2).
          const int row0 = e_row - lane;                      // this warp's first row within the sequence
          uint16_t* const base = (e_slot < 0 ? reinterpret_cast<uint16_t*>(prm.out) + (static_cast<size_t>(e_b) * prm.R + row0) * kDv
                                             : partial_halves(prm) + static_cast<size_t>(prow0 + (quarter & 1) * 32) * kDv) + col0;
          const uint32_t stage = smem_base + kOffP + (2 * khalf + grp) * kPPageBytes + (quarter & 1) * 32 * 128;
          uint32_t sc = 0;                                    // this thread's four scale bytes
#pragma unroll 1
          for (int c = 0; c < 4; c += 2) {
            uint32_t o[2][32];
            tmem_ld_32x32b_x32(o_addr + 32 * c, o[0]);
            tmem_ld_32x32b_x32(o_addr + 32 * (c + 1), o[1]);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              uint32_t w[16];
              if (e_slot < 0) epilogue_chunk_bf16(o[e], e_inv, w);
              else sc |= epilogue_chunk_partial(o[e], e_inv, w) << (8 * (c + e));
#pragma unroll
              for (int i = 0; i < 4; ++i) st_shared_v4(stage + sw128_offset(lane, 4 * e + i), w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int rr = 4 * i + (lane >> 3), piece = lane & 7;
              uint32_t x[4];
              ld_shared_v4(stage + sw128_offset(rr, piece), x[0], x[1], x[2], x[3]);
              if (row0 + rr < prm.R) stg_128(base + rr * kDv + 32 * c + 8 * piece, x[0], x[1], x[2], x[3]);
            }
            __syncwarp();
          }
          if (valid) {
            if (e_slot >= 0) *reinterpret_cast<uint32_t*>(partial_scales(prm) + static_cast<size_t>(prow0 + r) * 16 + col0 / 32) = sc;
            if (khalf == 0 && grp == 0) {
              if (e_slot < 0) prm.lse[static_cast<size_t>(e_b) * prm.R + e_row] = e_lse;
              else prm.part_lse[prow0 + r] = e_lse;
            }
          }
          e_row = -1;
          if (tid == 0 && leader) AMLA_STAMP(prm, part, 14, gs - 1);
          if (!tile.valid) break;
          group_sync();                                       // the row group's four warps are done with their rows of the P buffer
          if (!ok) break;
        } else if (moved) {
          // lines 13-16: O <- AS_FP32(AS_INT32(O) + N).  The guarded add costs four integer operations per element, the
          // FP32 multiply it replaces one.  The guard only matters for an element whose magnitude bits plus N would not
          // stay positive (an exact zero, a value about to leave the normal range); so the smallest magnitude of the chunk
          // is taken first (half an operation per element), and where it is safe the chunk gets the plain one-instruction
          // add of Lemma 3.1.
#pragma unroll 1
          for (int c = 0; c < 4; ++c) {
            uint32_t o[32];
            tmem_ld_32x32b_x32(o_addr + 32 * c, o);
            tmem_wait_ld();
            if (kMode == 2) {
#pragma unroll
              for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * __uint_as_float(nword));
            } else {
              bool safe = true;
              if (kGuard) {
                float lo = fmin3_abs(__uint_as_float(o[0]), __uint_as_float(o[1]), __uint_as_float(o[2]));
#pragma unroll
                for (int i = 3; i + 1 < 32; i += 2) lo = fmin3_abs(lo, __uint_as_float(o[i]), __uint_as_float(o[i + 1]));
                lo = fminf(lo, fabsf(__uint_as_float(o[31])));
                // NaN magnitudes compare as large numbers and take the plain add, like every other normal pattern
                safe = __float_as_int(lo) + static_cast<int>(nword) > 0;
              }
              if (safe) {
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(exponent_add_raw(__uint_as_float(o[i]), static_cast<int>(nword)));
              } else {
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(exponent_add_guarded(__uint_as_float(o[i]), static_cast<int>(nword)));
              }
            }
            tmem_st_32x32b_x32(o_addr + 32 * c, o);
          }
          tmem_wait_st();
        }
        if (tid == 0 && leader) AMLA_STAMP(prm, part, 11, gs);
#pragma unroll 1
        for (int h = 0; grp + 2 * h < np && h < 2; ++h) {
          uint32_t pk[16];
          tmem_ld_32x32b_x16(scol + 64 * h, pk);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 4; ++c) store_p_piece(chunk0 + 2 * h, c, pk);
        }
      }
      tc_fence_before_sync();            // S has been read, O (perhaps) rewritten
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        if (leader) { mbar_arrive(bar(X_SEMPTY + sb)); mbar_arrive(bar(X_PREADY)); }
        else {                             // P~ of the whole warp, for the MMA issuer in the other CTA
          release_shared_to_cluster();
          mbar_arrive_cluster_relaxed(lead_bars + 8u * (X_SEMPTY + sb));
          mbar_arrive_cluster_relaxed(lead_bars + 8u * X_PREADY);
        }
      }
      if (tid == 0 && leader) AMLA_STAMP(prm, part, 12, gs);
      ++gs;
      if (tile.last()) {                   // what the unit's epilogue needs
        const Unit& u = tile.u;
        int2 info;
        e_slot = tile.units.slot_of(u, &info);
        if (tid == 0 && leader) merge_note(prm, part, u.it, info);
        e_b = u.b;
        e_row = u.r0 + rank * kCtaRows + r;
        float l4[4];
        exchange(st.l, l4);
        if (!ok) break;
        const float l_all = (l4[0] + l4[1]) + (l4[2] + l4[3]);
        const bool live = l_all > 0.f;
        e_inv = live ? prm.out_scale / (l_all * st.s_out) : 0.f;
        e_lse = live ? (st.m2 + log2f(l_all)) * kLn2 : -INFINITY;
      }
      tile.next();
      if (wid == kAsksForQ && tile.valid && tile.first) look_ahead();
    }
    if (!ok && lane == 0) {
      report_timeout(prm.status);
      if (leader && q_asked > 0) mbar_wait(bar(X_QFULL), q_asked & 1);     // let copies that may still be in flight land
    }
  } else if (wid == 8 || (!kFp8 && wid >= 10)) {
    // ======================================================== TMA loads, in the order in which the MMAs use them:
    // K(0), K(1), V(0), K(2), V(1), ..., K(n-1), V(n-2), V(n-1), the tiles counted over all of the part's units.
    //   bf16: one ring of 16 KB slots carries K (one 64-column block of half the tile's keys) and V (one page x 128 columns).
    //     The loader warps walk the same sequence and issue every third load of it: a slot takes ~350 clk to issue.
    //     With each V load goes a request to bring an eighth of the next tile's K into L2.  A slot that waits for HBM turns
    //     around in ~3000 clk, and while the ring is full of V, which L2 has, nothing is under way from HBM: the next K comes
    //     from L2 by the time its turn in the ring is there.  32 x 4096 keys 56.3 -> 54.6 us, 96 x 2048 82.7 -> 81.0.  (The
    //     contiguous form: asked for by the tensor map's boxes 55.8.  A tile earlier: 55.9, 96 x 2048 82.5: V is gone from L2
    //     by the time it is wanted.  Rings for K and for V by themselves: 63-67, as either is too short for its latency.  V of
    //     a tile between the K blocks of the one two after it: 57.0, rising logits 93 -> 100, the last tiles' V comes later.)
    //     Four loaders -> three: 53.9 -> 53.7, 1 x 2531 12.65 -> 12.55, 1 x 1500 12.08 -> 11.89.  (Room for a merge block beside a
    //     decode CTA is not why: twelve warps of 152 registers leave 7168, and the smallest merge block takes 8192.)
    //   E4M3: the same, by one loader into the raw ring.
    if (elect_one()) {
      const uint64_t keep = l2_policy_evict_normal(), last_use = l2_policy_evict_first();   // K: V follows a tile later; V: done with
      // first key row of a page; E4M3: a page outside the cache reads as zeros (rows behind the end of the tensor do)
      auto row_of = [&](int page) { return (kFp8 && (page < 0 || page >= prm.num_blocks) ? prm.num_blocks : page) * kPage; };
      // The page numbers of a tile are loaded once, a tile ahead: a load of the block table in front of every slot cost a loader
      // 500 clk there (a tile of the E4M3 cache took 11.9 K clk instead of 10.4 K).
      auto take = [&](Pages& pg) {                          // on to the next tile: its pages, 0: there is none
        tile.next();
        pg = load_pages(prm, tile);
        return tile.valid ? tile.np : 0;
      };
      // This CTA's half of the tile's keys, 32 np of them from key 32 np rank on, is at most two boxes: a page, or the half page
      // in the middle of a tile of three pages or of one.  (With 32 keys of every page it was four boxes: E4M3, one loader:
      // 62.6 -> 61.2 us for 32 x 4096 keys, 120.1 -> 116.4 for 32 x 512-8192, two tokens; bf16 494 -> 481 for 96 x 16384.)
      struct KBoxes {
        const CUtensorMap *map0, *map1;
        int row0, row1, chunks0, chunks1;                   // in chunks of 32 keys
      };
      auto boxes = [&](int np, const Pages& pg) {
        KBoxes x;
        const bool odd = (np * rank) & 1;                                 // begins in the middle of a page
        x.chunks0 = odd || np == 1 ? 1 : 2; x.chunks1 = min(np - x.chunks0, 2);
        x.row0 = row_of(rank == 0 || np == 1 ? pg.a : np == 4 ? pg.c : pg.b) + (odd ? 32 : 0);
        x.row1 = row_of(rank == 0 ? pg.b : np == 4 ? pg.d : pg.c);
        x.map0 = x.chunks0 == 2 ? &k_map : &khalf_map;
        x.map1 = x.chunks1 == 2 ? &k_map : &khalf_map;
        return x;
      };
      const uint32_t lead_full = lead_bars + 8u * X_FULL;
      if (wid == 8 && tile.valid)                           // the first unit's Q; the softmax warps ask for the others
        request_q(q_map, smem_base, bars, lead_bars, leader, q_row_of(prm, tile.u, rank));
      uint32_t n = 0;                                       // slots so far
      if constexpr (!kFp8) {
        const uint32_t mine = wid == 8 ? 0 : wid - 9;
        constexpr uint32_t kRing = kSlots<false>;
        uint32_t slot = 0, par = 1, turn = 0;
        auto advance = [&]() { if (++slot == kRing) { slot = 0; par ^= 1; } ++n; if (++turn == kLoaders) turn = 0; };
        Pages pg = first_pages, pg_nxt = {}, pg_prev = {};
        int np = tile.valid ? tile.np : 0, np_prev = 0;
        KBoxes x = boxes(np, pg);
        while (ok && np > 0) {
          int np_nxt = 0;
#pragma unroll 1
          for (int c = 0; c < kQBlocks; ++c) {
            if (c == kLoaders) np_nxt = take(pg_nxt);       // (behind this loader's first load: at a call's start that one is waited for)
            if (turn == mine) {
              ok = mbar_wait(bar(X_EMPTY) + 8 * slot, par);
              if (!ok) break;
              const uint32_t dst = smem_base + kOffRing + slot * kSlotBytes;
              if (leader) mbar_arrive_expect_tx(bar(X_FULL) + 8 * slot, 2 * np * kKBoxBytes);
              tma_load_3d_pair_hint(dst, x.map0, 0, x.row0, c, lead_full + 8 * slot, keep);
              if (x.chunks1 > 0) tma_load_3d_pair_hint(dst + x.chunks0 * kKBoxBytes, x.map1, 0, x.row1, c, lead_full + 8 * slot, keep);
            }
            advance();
          }
          x = boxes(np_nxt, pg_nxt);
          // V of the tile before (whatever unit that was in), and behind the part's last K its own V
          for (int k = 0; k < (np_nxt > 0 ? 1 : 2) && ok; ++k) {
            const int np_v = k == 0 ? np_prev : np;
            if (k > 0) pg_prev = pg;
#pragma unroll 1
            for (int i = 0; i < 2 * np_v; ++i) {
              if (turn == mine) {
                ok = mbar_wait(bar(X_EMPTY) + 8 * slot, par);
                if (!ok) break;
                if (leader) mbar_arrive_expect_tx(bar(X_FULL) + 8 * slot, 2 * kSlotBytes);
                tma_load_3d_pair_hint(smem_base + kOffRing + slot * kSlotBytes, &v_map, 0, pg_prev.a * kPage, 4 * rank + 2 * (i & 1), lead_full + 8 * slot, last_use);
                if (i < 2 * np_nxt) {                       // 16 rows of this CTA's half of the next tile's keys
                  const int row = (i < 2 * x.chunks0 ? x.row0 : x.row1 - 32 * x.chunks0) + 16 * i;
                  if (static_cast<uint32_t>(row) < static_cast<uint32_t>(prm.num_blocks * kPage)) bulk_prefetch_l2(prm.kv + static_cast<size_t>(row) * kDqk, 16 * kDqk * 2);
                }
              }
              if (i & 1) { pg_prev.a = pg_prev.b; pg_prev.b = pg_prev.c; pg_prev.c = pg_prev.d; }
              advance();
            }
          }
          np_prev = np; pg_prev = pg;
          np = np_nxt; pg = pg_nxt;
        }
        if (!ok) {
          report_timeout(prm.status);
          // let the copies that may still be in flight land before the CTA exits
          for (uint32_t i = 0; i < kRing && i < n; ++i) {
            const uint32_t k = n - 1 - i;
            if (leader && k % kLoaders == mine) mbar_wait(bar(X_FULL) + 8 * (k % kRing), (k / kRing) & 1);
          }
        }
      } else {
        uint32_t slot = 0, par = 1;
        auto advance = [&]() { if (++slot == kRawSlots) { slot = 0; par ^= 1; } ++n; };
        Pages pg = first_pages, pg_nxt = {}, pg_prev = {};
        int np = tile.valid ? tile.np : 0, np_prev = 0;
        while (ok && np > 0) {
          int np_nxt = 0;
          const KBoxes x = boxes(np, pg);
          // a raw slot is two column blocks of K (the last one by itself: its box reaches past the row's end, where there are zeros
          // that nothing reads), or a page of V, this CTA's 256 columns of it
#pragma unroll 1
          for (int c = 0; c < kQBlocks; c += 2) {
            if (c == 2) np_nxt = take(pg_nxt);
            const uint32_t full = bar(X_RAWFULL) + 8 * slot, dst = smem_base + kOffRaw + slot * kRawBytes;
            ok = mbar_wait(bar(X_RAWEMPTY) + 8 * slot, par);
            if (!ok) break;
            mbar_arrive_expect_tx(full, np * kKBoxBytes);
            tma_load_2d_hint(dst, x.map0, 64 * c, x.row0, full, keep);                                          // [64 or 32 keys][128 columns]
            if (x.chunks1 > 0) tma_load_2d_hint(dst + x.chunks0 * kKBoxBytes, x.map1, 64 * c, x.row1, full, keep);
            advance();
          }
          // V of the tile before (whatever unit that was in), and behind the part's last K its own V
          for (int k = 0; k < (np_nxt > 0 ? 1 : 2) && ok; ++k) {
            if (k > 0) pg_prev = pg;
#pragma unroll 1
            for (int i = k == 0 ? np_prev : np; i > 0; --i) {
              const uint32_t full = bar(X_RAWFULL) + 8 * slot;
              ok = mbar_wait(bar(X_RAWEMPTY) + 8 * slot, par);
              if (!ok) break;
              mbar_arrive_expect_tx(full, kRawBytes);
              tma_load_2d_hint(smem_base + kOffRaw + slot * kRawBytes, &v_map, 256 * rank, row_of(pg_prev.a), full, last_use);   // [64 keys][256 columns]
              pg_prev.a = pg_prev.b; pg_prev.b = pg_prev.c; pg_prev.c = pg_prev.d;
              advance();
            }
          }
          np_prev = np; pg_prev = pg;
          np = np_nxt; pg = pg_nxt;
        }
        if (!ok) {
          report_timeout(prm.status);
          for (uint32_t i = 0; i < kRawSlots && i < n; ++i) mbar_wait(bar(X_RAWFULL) + 8 * ((n - 1 - i) % kRawSlots), ((n - 1 - i) / kRawSlots) & 1);
        }
      }
      if (!ok && leader && wid == 8) mbar_wait(bar(X_QFULL), 0);
    }
    __syncwarp();
  } else if (kFp8 && wid >= 10) {
    // ======================================================== E4M3 cache: raw slot -> operand slots.  The three pairs of
    // warps take every third operand slot each; a thread widens 16 bytes at a time (exact: E4M3 values are bf16 values)
    // and stores them where the 128-byte swizzle of the operand tiles puts them.  (Raw slots of two operand slots: nine loads
    // a tile instead of seventeen, of which one loader had its hands full; and no bank conflicts, which V's stores had: 32 x 4096
    // keys 61.1 -> 60.5 us, 32 x 512-8192 with two tokens 122.2 -> 120.1.)
    const uint32_t mine = (wid - 10) / kWidenWarps;
    const int wt = ((wid - 10) % kWidenWarps) * 32 + lane;
    // `n` is the number of the slot, `pos` its place in the present phase (K of a tile: nine slots; V of one: two per page).
    // Two operand slots come from one raw slot, a tile's last block of K from one of its own.
    uint32_t n = mine, pos = mine, len = kQBlocks, raw_phase = 0;     // raw_phase: raw slots before this phase
    int np_prev = 0;                                     // pages of the tile before
    int what = tile.valid ? 0 : 3;                       // 0: K of the tile, 1: V of the tile before, 2: V of the part's last tile, 3: done
    while (ok) {
      while (pos >= len && what != 3) {                  // next phase
        pos -= len;
        raw_phase += (len + 1) >> 1;
        if (what == 0 && np_prev > 0) { what = 1; len = 2 * np_prev; }
        else if (what == 2) what = 3;
        else {
          np_prev = tile.np;
          tile.next();
          if (tile.valid) { what = 0; len = kQBlocks; }
          else { what = 2; len = 2 * np_prev; }
        }
      }
      if (what == 3) break;
      const bool is_k = what == 0;
      const uint32_t nth = raw_phase + (pos >> 1), second = pos & 1;
      const uint32_t rslot = nth % kRawSlots, rpar = (nth / kRawSlots) & 1;
      const uint32_t slot = n % kSlots<kFp8>, par = ((n / kSlots<kFp8>) & 1) ^ 1;
      // In this order.  Operand slot n is free: the MMAs have read number n - 4, and the raw slot in whose place this one stands
      // held numbers up to n - 4 at most, so it had been full.  (The other way round the wait for the raw slot could be let through
      // by the phase before that one's, when V has overtaken K.)
      ok = warp_wait(bar(X_EMPTY + slot), par);
      if (ok) ok = warp_wait(bar(X_RAWFULL + rslot), rpar);
      if (!ok) break;
      // Four threads take 64 columns of a row.  The eight that access shared memory together are placed so that no two of them
      // meet in a bank, neither in the load nor in the stores (whose rows alternate by the 128-byte swizzle):
      //   K: raw rows of two blocks, 128 bytes, swizzled likewise, row = page * 32 + key (rows of pages that the tile does not
      //      have hold older bytes; the MMA does not read them).  Rows a and a ^ 5: the other half of the banks in the raw
      //      slot, odd against even in the operand slot.
      //   V: raw rows of 256 bytes, 128 of them for this operand slot, 64 for each of its two blocks of 64 columns.  Rows a and
      //      a + 1 and different blocks.
      const uint32_t raw = smem_base + kOffRaw + rslot * kRawBytes, out = smem_base + kOffRing + slot * kSlotBytes;
      const int other = (wt >> 2) & 1, vblock = is_k ? 0 : ((wt >> 3) & 1) ^ other;
      const int r0 = is_k ? 8 * (wt >> 5) + (((wt >> 3) & 3) ^ (5 * other)) : 2 * (wt >> 4) + other;
      const uint32_t step = is_k ? 16 * 128 : 8 * 128;    // rows of a thread differ by multiples of 8: the same swizzle
      const uint32_t src = raw + (is_k ? r0 * 128 + (((4 * second + (wt & 3)) ^ (r0 & 7)) << 4) : r0 * 256 + 128 * second + 64 * vblock + 16 * (wt & 3));
      const uint32_t ch = 2 * (wt & 3), sw = r0 & 7;
      const uint32_t d0 = out + vblock * kVBlockBytes + r0 * 128 + ((ch ^ sw) << 4);
      const uint32_t d1 = (((ch + 1) ^ sw) << 4) - ((ch ^ sw) << 4);
      // Eight pieces of 16 bytes, all requested before the first is widened (four at a time: 32 x 4096 keys 58.0 us, so 56.9; 32 x
      // 512-8192 with two tokens 113.5 -> 111.3).  The raw slot is handed back at the end and not here: an arrival does not wait
      // for loads whose data nobody has used yet, and the next load by TMA then overtook them.
      uint32_t x[8][4];
#pragma unroll
      for (int k = 0; k < 8; ++k) ld_shared_v4(src + k * 2048, x[k][0], x[k][1], x[k][2], x[k][3]);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        uint32_t w[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) { w[2 * q] = e4m3x2_to_bf16x2(x[k][q]); w[2 * q + 1] = e4m3x2_to_bf16x2(x[k][q] >> 16); }
        st_shared_v4(d0 + k * step, w[0], w[1], w[2], w[3]);
        st_shared_v4(d0 + d1 + k * step, w[4], w[5], w[6], w[7]);
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar((leader ? X_FULL : X_FULLODD) + slot));
        mbar_arrive(bar(X_RAWEMPTY + rslot));
        if (pos + 1 == len && second == 0) mbar_arrive(bar(X_RAWEMPTY + rslot));   // (a raw slot of one block)
      }
      pos += kWidenGroups;
      n += kWidenGroups;
    }
    if (!ok && lane == 0) report_timeout(prm.status);
  } else if (kFp8 && wid == 9 && !leader) {
    // ======================================================== E4M3 cache, odd CTA: passes on to the MMA issuer that a slot is
    // full.  (By the widening warps themselves, behind a fence for every slot, 32 x 4096 keys took 58.1 us instead of 57.3, 32
    // x 4000 with two tokens 101.4 instead of 99.8; 8 x 1000 17.4 instead of 17.6.  With arrivals that published nothing: 56.9,
    // 98.9 and 17.1.)  A slot is filled again when the MMAs have read it, so no phase can pass unseen.
    if (elect_one()) {
      uint32_t slot = 0, par = 0;
      while (ok && tile.valid) {
        for (int i = kQBlocks + 2 * tile.np; i > 0 && ok; --i) {
          ok = mbar_wait(bar(X_FULLODD) + 8 * slot, par);
          if (!ok) break;
          release_shared_to_cluster();
          mbar_arrive_cluster_relaxed(lead_bars + 8u * (X_FULL + slot));
          if (++slot == kSlots<kFp8>) { slot = 0; par ^= 1; }
        }
        if (ok) tile.next();
      }
      if (!ok) report_timeout(prm.status);
    }
    __syncwarp();
  } else if (leader && wid == 9) {
    // ======================================================== MMA issuer (even CTA, for the pair)
    if (elect_one()) {
      constexpr uint32_t idesc_pv = make_idesc_bf16(128, 256, false, true);
      constexpr uint32_t idesc_qk1 = make_idesc_bf16(128, 64, false, false);     // N = 64 per page
      constexpr uint32_t idesc_step = make_idesc_bf16(128, 128, false, false) - idesc_qk1;
      constexpr uint32_t dhi = smem_desc_hi_sw128(1024);
      const uint32_t qlo = smem_desc_lo(smem_base + kOffQ, 16);
      const uint32_t plo = smem_desc_lo(smem_base + kOffP, 16);
      const uint32_t klo = smem_desc_lo(smem_base + kOffRing, 16);
      const uint32_t vlo = smem_desc_lo(smem_base + kOffRing, kVBlockBytes);
      uint32_t slot = 0, par = 0;
      uint32_t gs = 0, gp = 0, un = 0;                      // score tiles, P~V tiles, units so far
      auto advance = [&]() { if (++slot == kSlots<kFp8>) { slot = 0; par ^= 1; } };
      int np_prev = 0;                                      // pages of the tile before, 0: there was none
      bool fresh_prev = false;                              // it was its unit's first
      while (ok && tile.valid) {
        const int np = tile.np;
        const bool first = tile.first;
        if (first) {
          ok = mbar_wait(bar(X_QFULL), un & 1);
          if (!ok) break;
          ++un;
        }
        {
          const uint32_t sb = gs & 1;
          AMLA_STAMP(prm, part, 0, gs);
          ok = mbar_wait<true>(bar(X_SEMPTY + sb), ((gs >> 1) & 1) ^ 1);
          if (!ok) break;
          tc_fence_after_sync();
          AMLA_STAMP(prm, part, 1, gs);
          const uint32_t d = tbase + kSCol + 128 * sb;
          const uint32_t idesc = idesc_qk1 + (np - 1) * idesc_step;
#pragma unroll 1
          for (int c = 0; c < kQBlocks; ++c) {
            // bf16: TMA data -> MMA operand, both async proxy, no fence needed; E4M3: the widening threads have fenced
            ok = mbar_wait<kFp8>(bar(X_FULL) + 8 * slot, par);
            if (!ok) break;
            if (c == 0) AMLA_STAMP(prm, part, 2, gs);
            const uint32_t kl = klo + slot * (kSlotBytes >> 4), ql = qlo + c * (kQBlockBytes >> 4);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_ss_pair(d, smem_desc_join(ql + 2 * kk, dhi), smem_desc_join(kl + 2 * kk, dhi), idesc, (c | kk) != 0 ? 1u : 0u);
            mma_commit_pair_multicast(bar(X_EMPTY) + 8 * slot, 3);
            advance();
          }
          if (!ok) break;
          mma_commit_pair_multicast(bar(X_SFULL + sb), 3);
          AMLA_STAMP(prm, part, 3, gs);
          ++gs;
        }
        tile.next();
        // O (+)= P~ V of the tile before, whatever unit that was in, and behind the part's last QK^T its own: per page two
        // N = 256 products (128 columns from either CTA)
        for (int k = np_prev == 0 ? 1 : 0; k < (tile.valid ? 1 : 2) && ok; ++k) {
          const int np_v = k == 0 ? np_prev : np;
          uint32_t acc = (k == 0 ? fresh_prev : first) ? 0u : 1u;
          AMLA_STAMP(prm, part, 4, gp);
          ok = mbar_wait<true>(bar(X_PREADY), gp & 1);
          if (!ok) break;
          AMLA_STAMP(prm, part, 5, gp);
          tc_fence_after_sync();               // the softmax warps may have rewritten O (tcgen05.st) before arriving
#pragma unroll 1
          for (int i = 0; i < 2 * np_v; ++i) {
            ok = mbar_wait<kFp8>(bar(X_FULL) + 8 * slot, par);
            if (!ok) break;
            if (i == 0) AMLA_STAMP(prm, part, 6, gp);
            const uint32_t pl = plo + (i >> 1) * (kPPageBytes >> 4), vl = vlo + slot * (kSlotBytes >> 4), d = tbase + kOCol + 128 * (i & 1);
            if (i >= 2) acc = 1u;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_ss_pair(d, smem_desc_join(pl + 2 * kk, dhi), smem_desc_join(vl + 128 * kk, dhi), idesc_pv, kk == 0 ? acc : 1u);
            mma_commit_pair_multicast(bar(X_EMPTY) + 8 * slot, 3);
            advance();
          }
          if (!ok) break;
          mma_commit_pair_multicast(bar(X_PVDONE), 3);
          AMLA_STAMP(prm, part, 7, gp);
          ++gp;
        }
        np_prev = np;
        fresh_prev = first;
      }
      if (!ok) report_timeout(prm.status);
    }
    __syncwarp();
  }

  if (tid == 0 && leader) AMLA_STAMP(prm, part, 20, 2);
  // teardown: nobody may still be signalling a CTA that has exited, and both CTAs must be done with tensor memory
  tc_fence_before_sync();
  __syncthreads();
  cluster_arrive();
  cluster_wait();
  if (wid == 9) tmem_dealloc_pair(tbase, kTmemCols);
}

// ---------------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------------
namespace {

template <int kMode, bool kGuard, bool kFp8>
cudaError_t launch_variant(const CUtensorMap& kmap, const CUtensorMap& khalf, const CUtensorMap& vmap, const CUtensorMap& qmap, const DecodeParams& prm, cudaStream_t stream) {
  static std::atomic<uint64_t> done{0};
  return launch_serialized(decode_pair_kernel<kMode, kGuard, kFp8>, done, 2 * prm.P, kThreads<kFp8>, kSmemBytes, stream, kmap, khalf, vmap, qmap, prm);
}

template <bool kFp8>
cudaError_t launch_mode(const CUtensorMap& kmap, const CUtensorMap& khalf, const CUtensorMap& vmap, const CUtensorMap& qmap, const DecodeParams& prm, cudaStream_t stream) {
  const int mode = prm.flags & 3;
  const bool guard = !(prm.flags & 4);
  if (mode == 0) return guard ? launch_variant<0, true, kFp8>(kmap, khalf, vmap, qmap, prm, stream) : launch_variant<0, false, kFp8>(kmap, khalf, vmap, qmap, prm, stream);
  if (mode == 1) return guard ? launch_variant<1, true, kFp8>(kmap, khalf, vmap, qmap, prm, stream) : launch_variant<1, false, kFp8>(kmap, khalf, vmap, qmap, prm, stream);
  return launch_variant<2, true, kFp8>(kmap, khalf, vmap, qmap, prm, stream);
}

// An E4M3 cache: rows of 576 bytes.
bool encode_bytes(EncodeTiledFn encode, CUtensorMap* map, const void* base, cuuint64_t rows, cuuint32_t box_rows, cuuint32_t box_cols, bool swizzle) {
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(kDqk), rows};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(kDqk)};
  const cuuint32_t box[2] = {box_cols, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Number of two-CTA clusters the schedule is cut into: one per SM pair.
int decode_pair_parts(int sm_count) { return sm_count / 2 > 0 ? sm_count / 2 : 1; }

cudaError_t launch_decode_pair(const DecodeParams& prm, cudaStream_t stream, int* unsupported) {
  *unsupported = 0;
  EncodeTiledFn encode = get_encode_fn();
  if (!encode) { *unsupported = 1; return cudaErrorNotSupported; }
  // K: a page or half of one (32 keys) x one column block; V: a page x two column blocks; Q: a CTA's 64 rows x three column
  // blocks (rows past the end of the array read as zero, rows of a following sequence are computed and dropped)
  CUtensorMap kmap, khalf, vmap, qmap;
  const cuuint64_t keys = static_cast<cuuint64_t>(prm.num_blocks) * kPage;
  if (!encode_rows(encode, &qmap, prm.q, static_cast<cuuint64_t>(prm.B) * prm.R, kCtaRows, 3)) return cudaErrorInvalidValue;
  if (prm.kv8 != nullptr) {
    if (!encode_bytes(encode, &kmap, prm.kv8, keys, 64, 128, true) || !encode_bytes(encode, &khalf, prm.kv8, keys, 32, 128, true) ||
        !encode_bytes(encode, &vmap, prm.kv8, keys, 64, 256, false))
      return cudaErrorInvalidValue;
    return launch_mode<true>(kmap, khalf, vmap, qmap, prm, stream);
  }
  if (!encode_rows(encode, &kmap, prm.kv, keys, 64, 1) || !encode_rows(encode, &khalf, prm.kv, keys, 32, 1) || !encode_rows(encode, &vmap, prm.kv, keys, 64, 2)) return cudaErrorInvalidValue;
  return launch_mode<false>(kmap, khalf, vmap, qmap, prm, stream);
}

}  // namespace amla
