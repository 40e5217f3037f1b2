// How a cluster walks its share of the schedule: units (the part of one item that falls into the cluster's range) and,
// inside a unit, score tiles of a few 64-key pages.  Every role of a cluster runs the same walk, so no role has to tell
// another what comes next.  (Include after amla_common.cuh.)
#pragma once

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
template <bool kGuess>
__device__ __forceinline__ int load_length(const DecodeParams& prm, int b) {
  int n;
  if (kGuess) asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(n) : "l"(prm.seqlens + b) : "memory");
  else asm volatile("ld.global.b32 %0, [%1];" : "=r"(n) : "l"(prm.seqlens + b) : "memory");
  return min(max(n, 0), prm.max_blocks_per_seq * kPage);
}

// The schedule prefix of the batch, by one warp: into shared memory together with the sequence lengths (unless lens is null),
// or into the workspace.
//
// plan_on_chip also runs ahead of griddepcontrol.wait, when a kernel in front that produces the lengths may not have written
// them yet, or not so that this kernel sees it.  What it finds there is a guess, whatever it is: lengths are clamped to the
// table's width, for which the schedule's positions fit their type (the launch sees to that).  After the wait
// plan_is_stale() holds the guess against the lengths as they are; where they differ the plan is made again.
// (The guess is right unless the kernel directly in front writes the lengths.  One sequence of 256 keys with 16 heads: planned
// wholly behind the wait 8.5 us, guessed and checked 7.7, guessed and not checked 7.2; 32 x 4096 keys 51.7, 50.9 and 50.4,
// calls replayed back to back.)
__device__ __forceinline__ void plan_on_chip(const DecodeParams& prm, int* prefix, int* lens, int lane) {
  int carry = 0;
  for (int base = 0; base < prm.n_items; base += 32) {
    const int it = base + lane;
    const int b = prm.nrb == 1 ? it : it / prm.nrb;
    const int n_seq = it < prm.n_items ? load_length<true>(prm, b) : 0;
    const int v = it < prm.n_items ? schedule_length(n_seq, it, prm.tile_keys, prm.ovh) : 0;
    const int x = warp_inclusive_scan(v, lane);
    if (it < prm.n_items) {
      if (lens) lens[b] = n_seq;                         // same value from every row block
      prefix[it] = carry + x - v;
    }
    carry += __shfl_sync(0xffffffffu, x, 31);
  }
  if (lane == 0) prefix[prm.n_items] = carry;
}
// Page numbers of the first unit, on their way while the lengths are (the guess's place in the table is inside the table).
__device__ __forceinline__ void prefetch_pages(const DecodeParams& prm, int b, int page) {
  asm volatile("{\n\t.reg .b32 x;\n\tld.global.b32 x, [%0];\n\t}" ::"l"(prm.block_table + static_cast<size_t>(b) * prm.max_blocks_per_seq + page));
}
// By all threads of the CTA, after griddepcontrol.wait: does the plan differ from what the lengths give?
__device__ __forceinline__ bool plan_is_stale(const DecodeParams& prm, const int* prefix, const int* lens, int tid, int threads) {
  bool stale = false;
  for (int it = tid; it < prm.n_items; it += threads) {
    const int b = prm.nrb == 1 ? it : it / prm.nrb;
    const int n_seq = load_length<false>(prm, b);
    stale |= lens ? lens[b] != n_seq : prefix[it + 1] - prefix[it] != schedule_length(n_seq, it, prm.tile_keys, prm.ovh);
  }
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

struct UnitIter {
  const DecodeParams& prm;
  const int* prefix;
  const int* seqlens;
  int p, g, g1, share, parts;
  __device__ UnitIter(const DecodeParams& prm_, const int* prefix_, const int* seqlens_, int part) : prm(prm_), prefix(prefix_), seqlens(seqlens_), p(part) {
    start();
  }
  __device__ void start() {
    const Plan plan = Plan::make(prefix, prm.n_items, prm.P, prm.ovh, prm.min_share);
    share = plan.share; parts = plan.P;
    if (plan.L <= 0 || p >= plan.P) { g = g1 = 0; }
    else { g = plan.part_start(p); g1 = plan.part_start(p + 1); }
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
  __device__ explicit TileIter(const UnitIter& it) : units(it) { begin(); }
  __device__ bool last() const { return left == 0; }
  __device__ void begin() {
    valid = units.next(u);
    if (!valid) return;
    const int n = u.t1 - u.t0, nt = (n + kMaxPages - 1) / kMaxPages;
    base = static_cast<int>(static_cast<unsigned>(n) / static_cast<unsigned>(nt)); rem = n - base * nt;
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
    if (left == 0) begin();
    else { step(); first = false; }
  }
};

}  // namespace amla
