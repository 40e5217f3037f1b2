// Test aid: the merge kernel of the library by itself, on the leavings of a decode kernel that a test has made up.
#include <cstring>

#include "../paper_2509_25224_b200/csrc/amla_plan_combine.cu"

// One sequence of 16 query rows in 32-row items (FP32 partials), four parts.
extern "C" int merge_alone(int* status, int4* merge_info, float* part_lse, float* part_o, __nv_bfloat16* out, float* lse, void* stream) {
  amla::DecodeParams prm;
  std::memset(&prm, 0, sizeof(prm));
  prm.status = status;
  prm.merge_info = merge_info;
  prm.part_lse = part_lse;
  prm.part_o = part_o;
  prm.out = out;
  prm.lse = lse;
  prm.B = prm.Sq = prm.nrb = prm.n_items = 1;
  prm.H = prm.R = 16;
  prm.P = 4;
  prm.sms = 148;
  prm.item_rows = 32;
  return amla::launch_combine(prm, static_cast<cudaStream_t>(stream)) == cudaSuccess ? 0 : -4;
}
