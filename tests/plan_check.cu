// Test aid: the check of a schedule on chip against the lengths as they are (amla_units.cuh), on the host.
#include "amla_units.cuh"

extern "C" int item_is_stale(int nrb, int tile_keys, int ovh, const int* prefix, const int* lens, const int* first_unit, int it, int n_seq) {
  amla::DecodeParams prm = {};
  prm.nrb = nrb;
  prm.tile_keys = tile_keys;
  prm.ovh = ovh;
  amla::FirstUnit first = {};
  first.u.it = first_unit[0];
  first.u.t0 = first_unit[1];
  first.u.t1 = first_unit[2];
  first.u.n_b = first_unit[3];
  return amla::item_is_stale(prm, prefix, lens, &first, it, n_seq) ? 1 : 0;
}
