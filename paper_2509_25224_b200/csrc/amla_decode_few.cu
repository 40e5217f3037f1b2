// Tensor-core MLA decode kernel for sequences of up to 32 query rows (16 heads of a model sharded by heads, say), sm_100a.
//
// With so few rows the call is a stream of the cache through the GPU; the kernel is built to load every page ONCE, to keep
// as many bytes on their way as shared memory holds, and to leave the tensor pipe time to spare.  One CTA works on all rows
// of a sequence and a range of its 64-key pages; three pages (221 KB) are its ring.
//
//   S = Q K^T       A = Q from tensor memory: the up to 32 rows repeated in each quarter of the 128 lanes, so that each of
//                   the four softmax warps (a warp reaches one quarter) has every row; B = the page, all 576 columns
//   O^T += V^T P~^T A = V^T: the SAME page in shared memory read along the other axis, 128 of V's columns at a time; B = P~
//                   (32 rows x 64 keys, shared memory).  With the product transposed V's columns fill the 128 lanes and
//                   the rows are N: 16 or 32, not 128 of which most would be padding
//
// Warps 0-3 run Algorithm 2's recurrence (lines 5-12).  A thread holds one row, takes the maximum over the page's 64 scores
// by itself and does the exponentials of 16 of them: no two threads have to agree on anything until the row sum is added
// up at the end.  They apply the integer N to the bit patterns of O when a row's reference moved (lines 13-16), run the
// epilogue (line 20), and lay Q out in tensor memory: for the next unit ahead of this unit's epilogue.  Warp 4 loads (TMA),
// warp 5 issues the QK^T products, warp 6 the P~V products.
//
// The 128-row kernel gives such sequences M = 128 products of which 16 rows count, loads the cache twice (K by halves of the
// keys, V by halves of the columns) and runs into the power limit.  Against it (sustained): 32 sequences of 1-8 K keys, 16
// rows 56.5 -> 37.9 us; 32 x 4096, 32 rows 52.4 -> 39.6; 96 x 2048, 16 rows 77 -> 47.8; 192 of 1-512 keys 36.5 -> 25.2;
// 96 x 16384 518 -> 313 (1.81 GB: 5.8 TB/s; 6.5 TB/s before the power limit bites).
// What bounds it: the cache's bytes while pages are under way (a page needs ~2100 clk of products and hand-offs against the
// 2900 that 73,728 bytes take at a 148th of 7.1 TB/s), plus ~10 us of start, epilogue and merge.
//
// All waits are bounded; on expiry the kernel records kStatusTimeout and unwinds.
#include "amla_common.cuh"
#include "amla_host.cuh"
#include "amla_sm100.cuh"
#include "amla_units.cuh"

namespace amla {

using namespace sm100;

namespace {

constexpr int kSoftmaxWarps = 4;
constexpr int kLoadWarp = 4, kQkWarp = 5, kPvWarp = 6;
constexpr int kThreads = 32 * 7;
constexpr int kColBlocks = kDqk / 64;                   // 64-column blocks of a page
constexpr uint32_t kBlockBytes = kPage * 128;           // [64 keys][128 B], 128-byte swizzle
constexpr uint32_t kPageBytes = kColBlocks * kBlockBytes;
constexpr int kSlots = 3;                               // pages in shared memory
constexpr int kPieces = 3;                              // a page arrives in three pieces of three column blocks, a barrier each
constexpr uint32_t kPieceBytes = kPageBytes / kPieces;
constexpr uint32_t kQBlockBytes = kFewRows * 128;       // Q goes through a slot of the ring, too

constexpr uint32_t kOffP = kSlots * kPageBytes;         // P~: [32 rows][64 keys]
constexpr uint32_t kOffXchg = kOffP + kFewRows * 128;   // float [2][4 warps][32 rows]
constexpr uint32_t kOffBars = kOffXchg + 2 * kSoftmaxWarps * kFewRows * 4;
constexpr uint32_t kBarBytes = 256;
// a copy of the schedule prefix and of the sequence lengths for batches of up to kSmemPlanItems sequences
constexpr int kSmemPlanItems = 512;
constexpr uint32_t kOffPlan = kOffBars + kBarBytes;
constexpr uint32_t kOffSeqlens = kOffPlan + ((kSmemPlanItems + 1) * 4 + 15) / 16 * 16;
constexpr uint32_t kOffFirst = kOffSeqlens + kSmemPlanItems * 4;
constexpr uint32_t kSmemBytes = kOffFirst + sizeof(FirstUnit);
static_assert(kSmemBytes <= 232448, "exceeds the shared memory a block can opt in to");
static_assert(kPageBytes % 1024 == 0 && kOffP % 1024 == 0, "swizzled tiles need 1024-byte alignment");

// tensor-memory columns
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kQCol = 0;                           // 288 columns: 576 bf16 per row
constexpr uint32_t kOCol = 288;                         // 4 x 16 or 32: block m holds columns 128 m + lane of O, a row per column
constexpr uint32_t kSCol = 416;                         // 64; up to 16 rows, where O is smaller, the 64 before them as well

enum { X_FULL = 0, X_EMPTY = X_FULL + kSlots * kPieces, X_QREADY = X_EMPTY + kSlots, X_SFULL, X_SEMPTY = X_SFULL + 2, X_PREADY = X_SEMPTY + 2, X_XCHG, X_NUM };
static_assert(X_NUM * 8 + 8 <= kBarBytes, "barrier area too small");

__device__ __forceinline__ void report_timeout(int* status) { atomicExch(status, kStatusTimeout); }
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity)); }

using Tiles = TileIter<1>;

}  // namespace

template <int kMode, bool kGuard>
__global__ void __launch_bounds__(kThreads, 1)
decode_few_kernel(const __grid_constant__ CUtensorMap kv_map, const __grid_constant__ CUtensorMap q_map, const DecodeParams prm) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t smem_base = smem_u32(smem_raw);
  const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
  const int part = blockIdx.x;
  if (tid == 0) AMLA_STAMP(prm, part, 20, 0);
  if (smem_base & 1023u) {   // the swizzled tiles assume a 1024-byte aligned window
    if (tid == 0) report_timeout(prm.status);
    return;
  }
  const uint32_t bars = smem_base + kOffBars;
  auto bar = [&](int i) { return bars + 8u * i; };
  const uint32_t tmem_slot = bars + kBarBytes - 8;

  // Set-up.  The schedule is worked out from the sequence lengths as they are found (held against the final ones after the
  // wait below): all threads bring them, or the load warp where they are few, and the load warp adds up.  Beside that the MMA warp
  // allocates tensor memory and one thread of a softmax warp initialises the barriers.
  const bool plan_here = prm.fused_plan && prm.n_items <= kSmemPlanItems;
  int* plan_smem = reinterpret_cast<int*>(smem_raw + kOffPlan);
  int* lens_smem = reinterpret_cast<int*>(smem_raw + kOffSeqlens);
  FirstUnit* first_smem = reinterpret_cast<FirstUnit*>(smem_raw + kOffFirst);
  const bool by_warp = prm.n_items <= kWarpPlanItems;
  if (plan_here && (!by_warp || wid == kLoadWarp)) plan_lengths(prm, plan_smem, lens_smem, by_warp ? lane : tid, by_warp ? 32 : kThreads);
  if (tid == 0) {
    for (int i = 0; i < kSlots * kPieces; ++i) mbar_init(bar(X_FULL + i), 1);
    for (int i = 0; i < kSlots; ++i) mbar_init(bar(X_EMPTY + i), 1);
    mbar_init(bar(X_QREADY), kSoftmaxWarps);
    for (int i = 0; i < 2; ++i) { mbar_init(bar(X_SFULL + i), 1); mbar_init(bar(X_SEMPTY + i), kSoftmaxWarps); }
    mbar_init(bar(X_PREADY), kSoftmaxWarps);
    mbar_init(bar(X_XCHG), kSoftmaxWarps);
    fence_mbar_init();
    prefetch_tensormap(&kv_map);
    prefetch_tensormap(&q_map);
  }
  if (wid == kQkWarp) { tmem_alloc(tmem_slot, kTmemCols); tmem_relinquish(); }
  if (plan_here) {
    if (by_warp) __syncwarp(); else __syncthreads();
    if (wid == kLoadWarp) plan_units(prm, plan_smem, lens_smem, first_smem, part, lane);
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tbase = ld_shared_b32(tmem_slot);

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
  int first_page = 0;                                        // the load warp's first page: on its way while the lengths are
  auto load_page = [&]() { if (wid == kLoadWarp && tile.valid) first_page = ldg_here(prm.block_table + static_cast<size_t>(tile.u.b) * prm.max_blocks_per_seq + tile.t); };
  if (!plan_here) {
    load_page();
  } else {
    // Launched with programmatic stream serialization: everything above ran while the kernel before this one on the stream
    // was still going; its results (the previous call's reads of the workspace among them) are complete after this wait.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    load_page();                                             // (the guess's place in the table is inside the table)
    if (plan_is_stale(prm, plan_smem, lens_smem, first_smem, tid, kThreads)) {
      plan_lengths(prm, plan_smem, lens_smem, tid, kThreads);
      __syncthreads();
      if (wid == kLoadWarp) plan_units(prm, plan_smem, lens_smem, first_smem, part, lane);
      __syncthreads();
      tile.start(first_smem);
      load_page();
    }
    if (blockIdx.x == 0 && wid == 0 && lane == 0) *prm.status = kStatusOk;
  }
  if (tid == 0) AMLA_STAMP(prm, part, 20, 4);
  const bool wide = prm.R > 16;              // N of the P~V products: 16 or 32
  const uint32_t o_step = wide ? 32 : 16;    // tensor-memory columns per block of O
  const uint32_t s_two = wide ? 0 : 1;       // S is double buffered

  if (wid < kSoftmaxWarps) {
    // ======================================================== Q, softmax, correction, epilogue
    const int quarter = wid, r = lane;                   // thread = query row; the warp does keys 16 quarter .. + 15 of a page
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    const bool scale_nonneg = prm.scale_log2 >= 0.f;
    const uint32_t p_dst = smem_base + kOffP + r * 128, p_sw = r & 7;
    const uint32_t o_addr = tbase + lane_base + kOCol;
    const int halves_of_o = wide ? 2 : 1;
    uint32_t gs = 0, un = 0;
    uint32_t slot = 0, par = 0;                          // of the page (or Q) that comes next in the ring
    auto advance = [&]() { if (++slot == kSlots) { slot = 0; par ^= 1; } };
    // Copies the next unit's Q rows from their slot of the ring into this warp's quarter of tensor memory (rows that the
    // sequence does not have: zeros).
    auto load_q = [&]() {
      const uint32_t row = smem_base + slot * kPageBytes + r * 128;
      const uint32_t live = r < prm.R ? 1u : 0u;
#pragma unroll 1
      for (int p = 0; p < kPieces; ++p) {
        ok = warp_wait(bar(X_FULL + kPieces * slot + p), par);
        if (!ok) return;
        uint32_t w[3][32];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int i = 0; i < 8; ++i)
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\tmov.b32 %3, 0;\n\t"
                         "@p ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];\n\t}"
                         : "=&r"(w[c][4 * i]), "=&r"(w[c][4 * i + 1]), "=&r"(w[c][4 * i + 2]), "=&r"(w[c][4 * i + 3])
                         : "r"(row + (3 * p + c) * kQBlockBytes + ((i ^ p_sw) << 4)), "r"(live));
#pragma unroll
        for (int c = 0; c < 3; ++c) tmem_st_32x32b_x32(tbase + lane_base + kQCol + 32 * (3 * p + c), w[c]);
      }
      advance();
      tmem_wait_st();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(X_QREADY));
    };

    if (tile.valid) load_q();
    if (tid == 0) AMLA_STAMP(prm, part, 20, 1);
    if (tid == 0) merge_begin(prm, part);
    write_empty_items(prm, prefix, part, prm.P, 0, kFewRows, tid, 32 * kSoftmaxWarps);
    while (ok && tile.valid) {
      const Unit u = tile.u;
      const int visible = min(u.n_b, u.n_b - prm.Sq + r / prm.H + 1);  // keys 0..visible-1 are seen by this row
      const int first_masked = max(u.n_b - prm.Sq + 1, 0) / kPage;     // pages from here on may hold hidden keys
      RowState st;
      row_state_init(st);
      bool more = true;
      while (more) {
        const int t = tile.t;
        const uint32_t sb = gs & s_two, s_addr = tbase + lane_base + kSCol - 64 * (s_two - sb);
        ok = warp_wait(bar(X_SFULL + sb), (gs >> s_two) & 1);
        if (!ok) break;
        tc_fence_after_sync();
        if (tid == 0) AMLA_STAMP(prm, part, 8, gs);
        const bool plain = t < first_masked && scale_nonneg;             // every key of the page is visible
        // lines 5-6: running max, by every warp over all 64 keys
        uint32_t s[16];
        float tmax;
        {
          uint32_t v[32], w[32];
          tmem_ld_32x32b_x32(s_addr, v);
          tmem_ld_32x32b_x32(s_addr + 32, w);
          tmem_ld_32x32b_x16(s_addr + 16 * quarter, s);
          tmem_wait_ld();
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(X_SEMPTY + sb));  // the scores are in registers
          float a = -INFINITY, c = a;
          if (plain) {
#pragma unroll
            for (int i = 0; i < 32; i += 2) {
              a = fmax3(a, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
              c = fmax3(c, __uint_as_float(w[i]), __uint_as_float(w[i + 1]));
            }
            tmax = fmaxf(a, c) * prm.scale_log2;
          } else {
            const int nvis = visible - t * kPage;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              a = fmaxf(a, i < nvis ? __uint_as_float(v[i]) * prm.scale_log2 : -INFINITY);
              c = fmaxf(c, i + 32 < nvis ? __uint_as_float(w[i]) * prm.scale_log2 : -INFINITY);
            }
            tmax = fmaxf(a, c);
#pragma unroll
            for (int i = 0; i < 16; ++i)                   // scaled here; hidden keys become 2^-inf = 0
              s[i] = 16 * quarter + i < nvis ? __float_as_uint(__uint_as_float(s[i]) * prm.scale_log2) : 0xff800000u;
          }
        }
        // Lazy reference: when one row must move, every row whose maximum rose moves with it (moving early is always allowed);
        // the rows then tend to stay in step and O is rescaled on fewer pages.  The four warps hold the same rows and agree.
        const bool must = r < prm.R && tmax > st.m2 + prm.tau;             // (other lanes may hold anything)
        const RowStep sp = row_step<kMode>(st, tmax, __any_sync(0xffffffffu, must) ? 0.f : prm.tau);
        // Line 10's factor S16 goes into the exponential's argument; the row sum of line 6 is the sum of the same FP32 values,
        // taken before the bf16 cast and divided by S16 once per page.
        const float nsub = log2f_approx(sp.p_scale) - sp.m2_sub;
        const float sc = plain ? prm.scale_log2 : 1.f;
        const uint64_t sc2 = pack_f32x2(sc, sc), ns2 = pack_f32x2(nsub, nsub);
        uint64_t rs = pack_f32x2(0.f, 0.f);
        uint32_t pk[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float x0, x1;
          unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), sc2, ns2), x0, x1);
          const float q0 = ex2_approx(x0), q1 = ex2_approx(x1);
          rs = add_f32x2(rs, pack_f32x2(q0, q1));
          pk[i] = pack_bf16x2(q0, q1);
        }
        if (!tile.first) {
          // the P~V of the page before: it has read the P buffer, and O holds its sum
          ok = warp_wait(bar(X_EMPTY + (slot == 0 ? kSlots - 1 : slot - 1)), slot == 0 ? par ^ 1 : par);
          if (!ok) break;
          const uint32_t nword = (kMode == 2) ? __float_as_uint(sp.l_up) : static_cast<uint32_t>(sp.n_bits);
          const bool mine_moved = r < prm.R && ((kMode == 2) ? (sp.l_up != 1.f) : (sp.n_bits != 0));
          if (__any_sync(0xffffffffu, mine_moved)) {
            // lines 13-16: O <- AS_FP32(AS_INT32(O) + N).  O is transposed: a thread holds one column of O for 16 rows at a
            // time, and takes the rows' N from the lanes that hold the rows.
            tc_fence_after_sync();
#pragma unroll 1
            for (int h = 0; h < halves_of_o; ++h) {
              uint32_t nw[16];
#pragma unroll
              for (int i = 0; i < 16; ++i) nw[i] = __shfl_sync(0xffffffffu, nword, 16 * h + i);
#pragma unroll 1
              for (int m = 0; m < 4; ++m) {
                uint32_t o[16];
                tmem_ld_32x32b_x16(o_addr + o_step * m + 16 * h, o);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  const float f = __uint_as_float(o[i]);
                  o[i] = __float_as_uint(kMode == 2 ? f * __uint_as_float(nw[i])
                                         : kGuard   ? exponent_add_guarded(f, static_cast<int>(nw[i]))
                                                    : exponent_add_raw(f, static_cast<int>(nw[i])));
                }
                tmem_st_32x32b_x16(o_addr + o_step * m + 16 * h, o);
              }
            }
            tmem_wait_st();
          }
        }
        st_shared_v4(p_dst + (((2 * quarter) ^ p_sw) << 4), pk[0], pk[1], pk[2], pk[3]);
        st_shared_v4(p_dst + (((2 * quarter + 1) ^ p_sw) << 4), pk[4], pk[5], pk[6], pk[7]);
        tc_fence_before_sync();            // O (perhaps) rewritten
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(X_PREADY));
        if (tid == 0) AMLA_STAMP(prm, part, 12, gs);
        {
          float s0, s1;
          unpack_f32x2(rs, s0, s1);
          st.l = st.l * sp.l_up + __fdividef(s0 + s1, sp.p_scale);   // this warp's share of the row sum
        }
        ++gs;
        advance();
        more = !tile.last();
        if (more) tile.next();
      }
      if (!ok) break;
      // the next unit's Q: all QK^T of this one have been waited for
      const uint32_t last_slot = slot == 0 ? kSlots - 1 : slot - 1, last_par = slot == 0 ? par ^ 1 : par;
      tile.next();
      if (tile.valid) load_q();
      if (tid == 0) AMLA_STAMP(prm, part, 15, gs - 1);
      // ---- epilogue (line 20): out = O / (l * S16), lse = m + ln l
      if (!ok) break;
      int2 info;
      const int pslot = tile.units.slot_of(u, &info);      // partial slot, or -1
      if (tid == 0) merge_note(prm, part, u.it, info);
      const uint32_t xbuf = smem_base + kOffXchg + (un & 1) * (kSoftmaxWarps * kFewRows * 4) + r * 4;
      st_shared_b32(xbuf + quarter * (kFewRows * 4), __float_as_uint(st.l));
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(X_XCHG));
      ok = warp_wait(bar(X_XCHG), un & 1);
      if (!ok) break;
      ++un;
      float l_all = 0.f;
#pragma unroll
      for (int i = 0; i < kSoftmaxWarps; ++i) l_all += __uint_as_float(ld_shared_b32(xbuf + i * (kFewRows * 4)));
      const bool live = l_all > 0.f;
      const float inv = live ? prm.out_scale / (l_all * st.s_out) : 0.f;
      const float lse = live ? (st.m2 + log2f(l_all)) * kLn2 : -INFINITY;
      const size_t prow0 = static_cast<size_t>(pslot < 0 ? 0 : pslot) * kFewRows;    // first row of the partial arrays
      if (quarter == 0 && r < prm.R) {
        if (pslot < 0) prm.lse[static_cast<size_t>(u.b) * prm.R + r] = lse;
        else prm.part_lse[prow0 + r] = lse;
      }
      ok = warp_wait(bar(X_EMPTY + last_slot), last_par);
      if (!ok) break;
      tc_fence_after_sync();
      if (tid == 0) AMLA_STAMP(prm, part, 13, gs - 1);
      // A warp holds 32 neighbouring columns, one per lane: 64 bytes of a bf16 row or 128 of an FP32 partial per store.
      __nv_bfloat16* dst = prm.out + static_cast<size_t>(u.b) * prm.R * kDv + 32 * quarter + lane;
      float* pdst = prm.part_o + prow0 * kDv + 32 * quarter + lane;
#pragma unroll 1
      for (int h = 0; h < halves_of_o; ++h) {
        float iv[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) iv[i] = __shfl_sync(0xffffffffu, inv, 16 * h + i);
        const int rows = prm.R - 16 * h;
#pragma unroll 1
        for (int m = 0; m < 4; ++m) {
          uint32_t o[16];
          tmem_ld_32x32b_x16(o_addr + o_step * m + 16 * h, o);
          tmem_wait_ld();
          if (pslot < 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (i < rows) dst[i * kDv] = __float2bfloat16_rn(__uint_as_float(o[i]) * iv[i]);
          } else {                                           // rows that the sequence does not have: a slot has room for them
#pragma unroll
            for (int i = 0; i < 16; ++i) pdst[i * kDv] = __uint_as_float(o[i]) * iv[i];
          }
          dst += 128;
          pdst += 128;
        }
        dst += 16 * kDv - 512;
        pdst += 16 * kDv - 512;
      }
      tc_fence_before_sync();      // O has been read: this warp's next PREADY arrival lets the next unit overwrite it
      if (tid == 0) AMLA_STAMP(prm, part, 14, gs - 1);
    }
    if (!ok && lane == 0) report_timeout(prm.status);
  } else if (wid == kLoadWarp) {
    // ======================================================== TMA loads: pages in order
    if (elect_one()) {
      uint32_t slot = 0, par = 1, n_issued = 0;
      auto entry = [&]() { return prm.block_table + static_cast<size_t>(tile.u.b) * prm.max_blocks_per_seq + tile.t; };
      int page = first_page;
      auto load = [&](const CUtensorMap* map, int row, uint32_t piece_bytes) {
        ok = mbar_wait(bar(X_EMPTY) + 8 * slot, par);
        if (!ok) return;
        AMLA_STAMP(prm, part, 16, n_issued);
        const uint32_t dst = smem_base + slot * kPageBytes, full = bar(X_FULL) + 8 * kPieces * slot;
#pragma unroll
        for (int i = 0; i < kPieces; ++i) {
          mbar_arrive_expect_tx(full + 8 * i, piece_bytes);
          tma_load_3d(dst + i * piece_bytes, map, 0, row, kColBlocks / kPieces * i, full + 8 * i);
        }
        ++n_issued;
        if (++slot == kSlots) { slot = 0; par ^= 1; }
      };
      while (tile.valid) {
        if (tile.first) load(&q_map, tile.u.b * prm.R, kQBlockBytes * (kColBlocks / kPieces));
        if (!ok) break;
        const int row = page * kPage;
        tile.next();
        if (tile.valid) page = __ldg(entry());               // on its way while this page waits for its slot
        load(&kv_map, row, kPieceBytes);
        if (!ok) break;
      }
      if (!ok) {
        report_timeout(prm.status);
        // let the copies that may still be in flight land before the CTA exits
        for (uint32_t i = 0; i < kSlots && i < n_issued; ++i) {
          const uint32_t k = n_issued - 1 - i;
          for (int j = 0; j < kPieces; ++j) mbar_wait(bar(X_FULL) + 8 * (kPieces * (k % kSlots) + j), (k / kSlots) & 1);
        }
      }
    }
    __syncwarp();
  } else if (wid == kQkWarp) {
    // ======================================================== S = Q K^T.  (A warp for each of the two products: neither
    // waits behind the other's barriers, and together they keep the tensor pipe fed although either issues one page at a time.)
    if (elect_one()) {
      // up to 16 rows: M = 64, whose rows 16 i .. 16 i + 15 are lanes 32 i .. 32 i + 15 of tensor memory
      const uint32_t idesc = wide ? make_idesc_bf16(128, kPage, false, false) : make_idesc_bf16(64, kPage, false, false);
      constexpr uint32_t dhi = smem_desc_hi_sw128(1024);
      const uint32_t klo = smem_desc_lo(smem_base, 16);
      uint32_t slot = 0, par = 0, gs = 0, un = 0;
      auto advance = [&]() { if (++slot == kSlots) { slot = 0; par ^= 1; } };
      while (tile.valid) {
        if (tile.first) {
          ok = mbar_wait(bar(X_QREADY), un & 1);
          if (!ok) break;
          ++un;
          mbar_arrive(bar(X_EMPTY) + 8 * slot);              // Q has left its slot
          advance();
        }
        const uint32_t sb = gs & s_two, d = tbase + kSCol - 64 * (s_two - sb);
        ok = mbar_wait(bar(X_SEMPTY) + 8 * sb, ((gs >> s_two) & 1) ^ 1);
        if (!ok) break;
        tc_fence_after_sync();
        AMLA_STAMP(prm, part, 1, gs);
        uint32_t kl = klo + slot * (kPageBytes >> 4), qa = tbase + kQCol, acc = 0;
#pragma unroll 1
        for (int i = 0; i < kPieces; ++i) {                  // TMA data -> MMA operand, both async proxy, no fence needed
          ok = mbar_wait(bar(X_FULL) + 8 * (kPieces * slot + i), par);
          if (!ok) break;
          if (i == 0) AMLA_STAMP(prm, part, 2, gs);
#pragma unroll
          for (int c = 0; c < kColBlocks / kPieces; ++c)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_ts(d, qa + 32 * c + 8 * kk, smem_desc_join(kl + c * (kBlockBytes >> 4) + 2 * kk, dhi), idesc, (c | kk) != 0 ? 1u : acc);
          acc = 1;
          kl += kPieceBytes >> 4;
          qa += 32 * (kColBlocks / kPieces);
        }
        if (!ok) break;
        mma_commit(bar(X_SFULL) + 8 * sb);
        AMLA_STAMP(prm, part, 3, gs);
        ++gs;
        advance();
        tile.next();
      }
      if (!ok) report_timeout(prm.status);
    }
    __syncwarp();
  } else if (wid == kPvWarp) {
    // ======================================================== O^T (+)= V^T P~^T
    if (elect_one()) {
      const uint32_t idesc = wide ? make_idesc_bf16(128, 32, true, false) : make_idesc_bf16(128, 16, true, false);
      constexpr uint32_t dhi = smem_desc_hi_sw128(1024);
      const uint32_t vlo = smem_desc_lo(smem_base, kBlockBytes);
      const uint32_t plo = smem_desc_lo(smem_base + kOffP, 16);
      uint32_t slot = 0, gp = 0;
      auto advance = [&]() { if (++slot == kSlots) slot = 0; };
      while (tile.valid) {
        if (tile.first) advance();                           // Q's slot
        ok = mbar_wait(bar(X_PREADY), gp & 1);               // the scores of this page were there, so the page is
        if (!ok) break;
        tc_fence_after_sync();                               // the softmax warps may have rewritten O (tcgen05.st) before arriving
        AMLA_STAMP(prm, part, 5, gp);
        const uint32_t acc = tile.first ? 0u : 1u;
        uint32_t vl = vlo + slot * (kPageBytes >> 4), d = tbase + kOCol;
#pragma unroll 1
        for (int m = 0; m < 4; ++m) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_ss(d, smem_desc_join(vl + 128 * kk, dhi), smem_desc_join(plo + 2 * kk, dhi), idesc, kk == 0 ? acc : 1u);
          d += o_step;
          vl += 2 * kBlockBytes >> 4;
        }
        mma_commit(bar(X_EMPTY) + 8 * slot);                 // for the loader, and for the softmax warps: P~ and O
        AMLA_STAMP(prm, part, 7, gp);
        ++gp;
        advance();
        tile.next();
      }
      if (!ok) report_timeout(prm.status);
    }
    __syncwarp();
  }

  tc_fence_before_sync();
  __syncthreads();
  if (wid == kQkWarp) tmem_dealloc(tbase, kTmemCols);
}

// ---------------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------------
namespace {

template <int kMode, bool kGuard>
cudaError_t launch_variant(const CUtensorMap& kvmap, const CUtensorMap& qmap, const DecodeParams& prm, cudaStream_t stream) {
  static std::atomic<uint64_t> done{0};
  return launch_serialized(decode_few_kernel<kMode, kGuard>, done, prm.P, kThreads, kSmemBytes, stream, kvmap, qmap, prm);
}

}  // namespace

cudaError_t launch_decode_few(const DecodeParams& prm, cudaStream_t stream, int* unsupported) {
  *unsupported = 0;
  EncodeTiledFn encode = get_encode_fn();
  if (!encode) { *unsupported = 1; return cudaErrorNotSupported; }
  CUtensorMap kvmap, qmap;        // a third of a page; a third of a unit's 32 rows (rows past the end of the array read as zero)
  if (!encode_rows(encode, &qmap, prm.q, static_cast<cuuint64_t>(prm.B) * prm.R, kFewRows, kColBlocks / kPieces)) return cudaErrorInvalidValue;
  if (!encode_rows(encode, &kvmap, prm.kv, static_cast<cuuint64_t>(prm.num_blocks) * kPage, kPage, kColBlocks / kPieces)) return cudaErrorInvalidValue;
  const int mode = prm.flags & 3;
  const bool guard = !(prm.flags & 4);
  if (mode == 0) return guard ? launch_variant<0, true>(kvmap, qmap, prm, stream) : launch_variant<0, false>(kvmap, qmap, prm, stream);
  if (mode == 1) return guard ? launch_variant<1, true>(kvmap, qmap, prm, stream) : launch_variant<1, false>(kvmap, qmap, prm, stream);
  return launch_variant<2, true>(kvmap, qmap, prm, stream);
}

}  // namespace amla
