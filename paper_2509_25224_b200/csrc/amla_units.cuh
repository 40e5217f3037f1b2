// How a cluster walks its share of the schedule: units (the part of one item that falls into the cluster's range) and,
// inside a unit, score tiles of a few 64-key pages.  Every role of a cluster runs the same walk, so no role has to tell
// another what comes next.
#pragma once

#include "amla_common.cuh"
#include "amla_sm100.cuh"

namespace amla {

__device__ __forceinline__ int warp_inclusive_scan(int v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// A sequence length, clamped to the table's width.  kGuess: as it stands in the GPU's common cache at this moment; the SM's own
// cache neither answers nor keeps it.  Otherwise an ordinary load, which griddepcontrol.wait is in front of (0.2-0.4 us less on
// the way to a call's first load than the other kind).
__device__ __forceinline__ int clamp_length(const DecodeParams& prm, int n) { return min(max(n, 0), prm.max_blocks_per_seq * kPage); }
template <bool kGuess>
__device__ __forceinline__ int load_length_raw(const DecodeParams& prm, int b) {
  int n;
  if (kGuess) asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(n) : "l"(prm.seqlens + b) : "memory");
  else asm volatile("ld.global.b32 %0, [%1];" : "=r"(n) : "l"(prm.seqlens + b) : "memory");
  return n;
}
template <bool kGuess>
__device__ __forceinline__ int load_length(const DecodeParams& prm, int b) { return clamp_length(prm, load_length_raw<kGuess>(prm, b)); }

struct Unit {
  int b, r0, n_b, t0, t1, it;      // sequence, first row of the row block, keys, tile range [t0, t1) of the schedule, item
};

// The next unit at or after position g of a range that ends at g1.  Not inlined: every role asks for units, but seldom,
// and what a cluster executes over and over has to stay small (a kernel of 144 KB of code, with this walk written out at
// a dozen places, spent hundreds of cycles per score tile on instruction fetches in every role).
struct UnitFound {
  Unit u;
  int g;                           // position behind the unit
};
static __device__ __noinline__ UnitFound find_unit(const int* prefix, const int* seqlens, int n_items, int nrb, int item_rows, int max_keys, int ovh, int g, int g1) {
  UnitFound f;
  f.u.t0 = f.u.t1 = 0;
  f.u.it = f.u.b = f.u.r0 = f.u.n_b = 0;
  while (g < g1) {
    int lo = 0, hi = n_items - 1;                 // the item that holds position g (zero-tile items are skipped automatically)
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (prefix[mid] <= g) lo = mid; else hi = mid - 1;
    }
    const int a = prefix[lo] + item_overhead(lo, ovh), e = prefix[lo + 1];
    const int first = max(g, a), last = min(e, g1);
    g = last;
    if (last > first) {
      f.u.it = lo; f.u.t0 = first - a; f.u.t1 = last - a;
      f.u.b = nrb == 1 ? lo : static_cast<int>(static_cast<unsigned>(lo) / static_cast<unsigned>(nrb));
      f.u.r0 = (lo - f.u.b * nrb) * item_rows;
      f.u.n_b = min(max(seqlens[f.u.b], 0), max_keys);
      break;
    }                                             // else: only overhead positions of this item fell into the range
  }
  f.g = g;
  return f;
}

// The first unit of a part and where the walk stands behind it: worked out with the plan, kept on chip for all roles.  (Looked
// up by every thread for itself once the plan was there, it was 0.9-1.3 us of a call's start.)
struct FirstUnit {
  Unit u;                          // t0 == t1: the part has none
  int g, g1, share;
};

// The schedule prefix of the batch and the part's first unit, on chip.  plan_lengths() by all threads of the CTA, then a barrier,
// then plan_units() by one warp, then a barrier: all lengths are on their way together, and one scan does.  (By one warp, 32
// lengths at a time and each 32 a memory round trip and a scan, the plan of 192 items took 6800 clk, of 32 1550; so 2750 and 2100
// with the first unit in it.  From a CTA's first instruction to its first load: 192 x 1-512 keys 16.0 K clk, so 6.5 K and the call
// 42.2 -> 39.0 us; 32 x 4096 8.0 K, so 6.0 K and 52.8 -> 52.1, since that one runs at the power limit.)
//
// Both also run ahead of griddepcontrol.wait, when a kernel in front that produces the lengths may not have written
// them yet, or not so that this kernel sees it.  What is found there is a guess, whatever it is: lengths are clamped to the
// table's width, for which the schedule's positions fit their type (the launch sees to that).  After the wait
// plan_is_stale() holds the guess against the lengths as they are; where they differ the plan is made again.
// (The guess is right unless the kernel directly in front writes the lengths.  One sequence of 256 keys with 16 heads: planned
// wholly behind the wait 8.5 us, guessed and checked 7.7, guessed and not checked 7.2; 32 x 4096 keys 51.7, 50.9 and 50.4,
// calls replayed back to back.)
// The loops over items stay rolled: written out four times they were code that a short call runs through once, cold (one sequence
// of 256 keys with 16 heads 8.16 us, rolled 8.04; the check behind the wait 1113 clk, rolled 990).
// Up to kWarpPlanItems items the one warp brings the lengths too, beside the other warps' set-up and without a barrier in between:
// 32 lengths are one load of a warp.  (By all threads / by one warp, us: one sequence of 256 keys with 16 heads 7.97 / 7.94, two
// tokens 1 x 256 10.59 / 10.54, 16 x 1-300 14.81 / 14.77.)
constexpr int kWarpPlanItems = 32;
// Leaves every item's schedule length in prefix[], and the lengths in lens[] (unless that is null).
__device__ __forceinline__ void plan_lengths(const DecodeParams& prm, int* prefix, int* lens, int tid, int threads) {
#pragma unroll 1
  for (int it = tid; it < prm.n_items; it += threads) {
    const int b = prm.nrb == 1 ? it : it / prm.nrb, n = load_length<true>(prm, b);
    if (lens) lens[b] = n;                               // (row blocks of a sequence may differ in a guess: see item_is_stale)
    prefix[it] = schedule_length(n, it, prm.tile_keys, prm.ovh);
  }
}
__device__ __forceinline__ void plan_units(const DecodeParams& prm, int* prefix, const int* lens, FirstUnit* first, int part, int lane) {
  const int per = (prm.n_items + 31) >> 5, it0 = lane * per, it1 = min(it0 + per, prm.n_items);     // a lane takes neighbouring items
  int sum = 0;
#pragma unroll 1
  for (int it = it0; it < it1; ++it) sum += prefix[it];
  const int upto = warp_inclusive_scan(sum, lane), before = upto - sum, total = __shfl_sync(0xffffffffu, upto, 31);
#pragma unroll 1
  for (int it = it0, at = before; it < it1; ++it) {
    const int v = prefix[it];
    prefix[it] = at;
    at += v;
  }
  if (lane == 0) prefix[prm.n_items] = total;
  __syncwarp();
  // the part's range of positions, as Plan has it
  const unsigned L = total, share = Plan::share_of(total, prm.P, prm.min_share);
  unsigned g = part * share;
  const unsigned g1 = min(g + share, L);
  // its first unit: of the last lane whose items begin at or before g
  int it = (31 - __clz(__ballot_sync(0xffffffffu, it0 < it1 && static_cast<unsigned>(before) <= g) | 1)) * per;
  Unit u = {};
  while (g < g1) {
    while (it + 1 < prm.n_items && static_cast<unsigned>(prefix[it + 1]) <= g) ++it;
    const unsigned a = prefix[it] + item_overhead(it, prm.ovh), e = prefix[it + 1], from = max(g, a), to = min(e, g1);
    g = to;
    if (to > from) {                                     // (else only overhead positions of this item are in the range)
      u.it = it; u.t0 = from - a; u.t1 = to - a;
      u.b = prm.nrb == 1 ? it : static_cast<int>(static_cast<unsigned>(it) / static_cast<unsigned>(prm.nrb));
      u.r0 = (it - u.b * prm.nrb) * prm.item_rows;
      u.n_b = lens ? lens[u.b] : load_length<true>(prm, u.b);
      break;
    }
  }
  if (lane == 0) {
    first->u = u;
    first->g = g; first->g1 = g1; first->share = share;
  }
}
// Does a plan's item `it` differ from what the n_seq keys of its sequence give?
// The length that is on chip says it all where a sequence is one item.  Where it is several, each of them has loaded the length for
// itself: while a kernel in front is writing it, prefix[] may have got the old one from one row block and the new one, which
// lens[] then holds, from another.  So what prefix[] has of the item is looked at too.
__host__ __device__ inline bool item_is_stale(const DecodeParams& prm, const int* prefix, const int* lens, const FirstUnit* first, int it, int n_seq) {
  if (lens != nullptr) {
    if (lens[prm.nrb == 1 ? it : it / prm.nrb] != n_seq) return true;
    if (prm.nrb == 1) return false;
  }
  const bool of_first = lens == nullptr && it == first->u.it && first->u.t1 > first->u.t0;      // (a part without a unit has no length to be wrong)
  return prefix[it + 1] - prefix[it] != schedule_length(n_seq, it, prm.tile_keys, prm.ovh) || (of_first && n_seq != first->u.n_b);
}
// By all threads of the CTA, after griddepcontrol.wait: does the plan differ from what the lengths give?
__device__ __forceinline__ bool plan_is_stale(const DecodeParams& prm, const int* prefix, const int* lens, const FirstUnit* first, int tid, int threads) {
  bool stale = false;
#pragma unroll 1
  for (int it = tid; it < prm.n_items; it += threads)
    stale |= item_is_stale(prm, prefix, lens, first, it, load_length<false>(prm, prm.nrb == 1 ? it : it / prm.nrb));
  return __syncthreads_or(stale);
}
__device__ __forceinline__ void plan_in_workspace(const DecodeParams& prm, int lane) {
  int* pw = const_cast<int*>(prm.prefix);
  int carry = 0;
  for (int base = 0; base < prm.n_items; base += 32) {
    const int it = base + lane;
    const int v = it < prm.n_items ? schedule_length(prm.seqlens[it / prm.nrb], it, prm.tile_keys, prm.ovh) : 0;
    const int x = warp_inclusive_scan(v, lane);
    if (it < prm.n_items) pw[it] = carry + x - v;
    carry += __shfl_sync(0xffffffffu, x, 31);
  }
  if (lane == 0) pw[prm.n_items] = carry;
}

struct UnitIter {
  const DecodeParams& prm;
  const int* prefix;
  const int* seqlens;
  int p, g, g1, share;
  __device__ UnitIter(const DecodeParams& prm_, const int* prefix_, const int* seqlens_, int part) : prm(prm_), prefix(prefix_), seqlens(seqlens_), p(part) {}
  // The part's first unit: from what plan_units() left, or looked up in the workspace's prefix (first == nullptr).
  __device__ void start(const FirstUnit* first, Unit& u) {
    if (first != nullptr) {
      u = first->u;
      g = first->g; g1 = first->g1; share = first->share;
    } else {
      const Plan plan = Plan::make(prefix, prm.n_items, prm.P, prm.ovh, prm.min_share);
      share = plan.share;
      if (plan.L <= 0 || p >= plan.P) { g = g1 = 0; }
      else { g = plan.part_start(p); g1 = plan.part_start(p + 1); }
      u.t0 = u.t1 = 0;
      next(u);
    }
  }
  __device__ bool next(Unit& u) {
    if (g >= g1) return false;
    const UnitFound f = find_unit(prefix, seqlens, prm.n_items, prm.nrb, prm.item_rows, prm.max_blocks_per_seq * kPage, prm.ovh, g, g1);
    u = f.u;
    g = f.g;
    return u.t1 > u.t0;
  }
  // Partial slot of the unit, -1 if its item lies in one part; *info = (slot of the item's first partial, partials)
  __device__ int slot_of(const Unit& u, int2* info) const {
    const int begin = prefix[u.it];
    const int p_first = static_cast<int>(static_cast<unsigned>(begin + item_overhead(u.it, prm.ovh)) / static_cast<unsigned>(share));
    const int p_last = static_cast<int>(static_cast<unsigned>(prefix[u.it + 1] - 1) / static_cast<unsigned>(share));
    const int slot_first = 2 * p_first + (begin > p_first * share ? 1 : 0);
    *info = make_int2(slot_first, p_last - p_first + 1);
    return p_first == p_last ? -1 : p == p_first ? slot_first : 2 * p;
  }
};

// Items without tiles have no unit: their output is zero and their lse -inf.  `who` of `step` writers takes every step-th
// item; within an item this writes rows [row0, row0 + nrows) of its block.
// (The function takes values: a reference would make every caller keep the kernel's parameters in local memory.)
static __device__ __noinline__ void write_empty_items_of(const int* prefix, int n_items, int nrb, int item_rows, int R, __nv_bfloat16* out, float* lse,
                                                         int4* merge_info, int who, int step, int row0, int nrows, int tid, int threads) {
  for (int it = who; it < n_items; it += step) {
    if (prefix[it + 1] > prefix[it]) continue;
    const int b = it / nrb, r0 = (it - b * nrb) * item_rows + row0;
    const int rows = min(nrows, R - r0);
    if (tid == 0 && row0 == 0 && merge_info != nullptr) merge_info[it] = make_int4(0, 0, 0, 0);
    const size_t first = static_cast<size_t>(b) * R + r0;
    uint4* dst = reinterpret_cast<uint4*>(out + first * kDv);
    for (int i = tid; i < rows * (kDv / 8); i += threads) dst[i] = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < rows; i += threads) lse[first + i] = -INFINITY;
  }
}
__device__ __forceinline__ void write_empty_items(const DecodeParams& prm, const int* prefix, int who, int step, int row0, int nrows, int tid, int threads) {
  write_empty_items_of(prefix, prm.n_items, prm.nrb, prm.item_rows, prm.R, prm.out, prm.lse, merge_by_item(prm) ? prm.merge_info : nullptr, who, step,
                       row0, nrows, tid, threads);
}

// What a part leaves for the combine kernel, by one thread: begin() first, then note() once per unit with what slot_of said.
__device__ __forceinline__ void merge_begin(const DecodeParams& prm, int part) {
  if (!merge_by_item(prm)) prm.merge_info[part] = make_int4(0, 0, 0, 0);
}
__device__ __forceinline__ void merge_note(const DecodeParams& prm, int part, int it, int2 info) {
  if ((info.x >> 1) == part && (merge_by_item(prm) || info.y > 1))      // the part in which the item begins speaks for it
    prm.merge_info[merge_by_item(prm) ? it : part] = make_int4(it, info.x, info.y, 0);
}

// The score tiles of a unit: its n pages in ceil(n / kMaxPages) tiles of nearly equal size, so that no unit ends with
// a one-page tile (an MMA of 64 keys takes two thirds of the time of one of 256).
template <int kMaxPages>
struct TileIter {
  UnitIter units;
  Unit u;
  int t, np;             // first page of the tile (within the item), pages in it
  int left, base, rem;   // tiles of the unit after this one, pages of the remaining tiles: base + 1 for `rem` of them, else base
  bool first;            // first tile of its unit
  bool valid;
  __device__ TileIter(const UnitIter& it, const FirstUnit* of_part) : units(it) { start(of_part); }
  __device__ bool last() const { return left == 0; }
  __device__ void start(const FirstUnit* of_part) {
    units.start(of_part, u);
    valid = u.t1 > u.t0;
    if (valid) begin();
  }
  __device__ void begin() {
    const int n = u.t1 - u.t0, nt = static_cast<int>(static_cast<unsigned>(n + kMaxPages - 1) / kMaxPages);
    base = kMaxPages;                                    // n / nt
#pragma unroll
    for (int i = 1; i < kMaxPages; ++i) if (base * nt > n) --base;
    rem = n - base * nt;
    left = nt; first = true;
    t = u.t0; np = 0;
    step();
  }
  __device__ void step() {
    t += np;
    np = base + (rem > 0 ? 1 : 0);
    --rem; --left;
  }
  __device__ void next() {
    if (left == 0) { valid = units.next(u); if (valid) begin(); }
    else { step(); first = false; }
  }
};

}  // namespace amla
