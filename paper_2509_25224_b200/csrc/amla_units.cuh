// How a cluster walks its share of the schedule: units (the part of one item that falls into the cluster's range) and,
// inside a unit, score tiles of a few 64-key pages.  Every role of a cluster runs the same walk, so no role has to tell
// another what comes next.  (Include after amla_common.cuh.)
#pragma once

namespace amla {

struct Unit {
  int b, r0, n_b, t0, t1, it;      // sequence, first row of the row block, keys, page range [t0, t1), item
};

struct UnitIter {
  const DecodeParams& prm;
  Plan plan;
  int p, g, g1;
  const int* seqlens;
  __device__ UnitIter(const DecodeParams& prm_, const int* prefix, const int* seqlens_, int part)
      : prm(prm_), plan(Plan::make(prefix, prm_.n_items, prm_.P, prm_.ovh)), p(part), seqlens(seqlens_) {
    if (plan.L <= 0 || p >= plan.P) { g = g1 = 0; }
    else { g = plan.part_start(p); g1 = plan.part_start(p + 1); }
  }
  __device__ bool next(Unit& u) {
    int it, a;
    while (true) {
      if (g >= g1) return false;
      it = plan.item_of_tile(g);
      a = plan.first_tile(it);
      const int e = plan.prefix[it + 1];
      const int lo = max(g, a), hi = min(e, g1);
      g = min(e, g1);
      if (hi > lo) { u.t0 = lo - a; u.t1 = hi - a; break; }   // else: only overhead positions of this item fell into the part
    }
    u.it = it;
    u.b = it / prm.nrb;
    u.r0 = (it - u.b * prm.nrb) * prm.item_rows;
    u.n_b = min(max(seqlens[u.b], 0), prm.max_blocks_per_seq * kPage);
    return true;
  }
  // Partial slot of the unit, -1 if its item lies in one part (several divisions: only the epilogue asks);
  // *info = what the combine needs to know about the item
  __device__ int slot_of(const Unit& u, int2* info) const {
    int p_first, p_last;
    const int nsplit = plan.item_parts(u.it, &p_first, &p_last);
    *info = make_int2(plan.slot_of(p_first, u.it, p_first), nsplit);
    return nsplit == 1 ? -1 : plan.slot_of(p, u.it, p_first);
  }
};

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
    base = n / nt; rem = n - base * nt;
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
