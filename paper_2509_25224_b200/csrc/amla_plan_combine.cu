// Split-KV schedule (prefix of tile counts per work item) and the lse-weighted combine of split
// partials.  Neither is in the paper: its kernel runs batch 96 on 48 cores, whereas a decode batch
// here has far fewer (sequence, row-block) items than the GPU has SMs.  The combine is the
// log-sum-exp merge that follows from the blockwise associativity of Algorithm 1's recurrence.
#include "amla_common.cuh"

namespace amla {

// One block.  prefix[it] = sum over items before `it` of their schedule lengths (tiles plus the start-up
// overhead of a non-empty item, see Plan); also resets the
// status word.  n_items is small (B * ceil(Sq*H/128)); a chunked block scan covers any size.
__global__ void plan_kernel(const int32_t* __restrict__ seqlens, int nrb, int n_items, int tile_keys, int ovh,
                            int* __restrict__ prefix, int* __restrict__ status) {
  __shared__ int warp_sums[32];
  __shared__ int carry;
  asm volatile("griddepcontrol.launch_dependents;");   // the decode kernel may start its set-up; it waits before reading
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) { carry = 0; *status = kStatusOk; }
  __syncthreads();
  for (int base = 0; base < n_items; base += blockDim.x) {
    const int it = base + tid;
    int v = 0;
    if (it < n_items) v = schedule_length(seqlens[it / nrb], it, tile_keys, ovh);
    int x = v;  // inclusive warp scan
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
      int s = (lane < (blockDim.x >> 5)) ? warp_sums[lane] : 0;
      for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
      }
      warp_sums[lane] = s;  // inclusive over warps
    }
    __syncthreads();
    const int before = carry + (wid ? warp_sums[wid - 1] : 0) + (x - v);
    if (it < n_items) prefix[it] = before;
    __syncthreads();
    if (tid == blockDim.x - 1) carry = before + v;
    __syncthreads();
  }
  if (tid == 0) prefix[n_items] = carry;
}

// The merge of split items,
//   lse = ln sum_s exp(lse_s),  out = sum_s exp(lse_s - lse) * out_s.
// The decode kernel left in merge_info which items are split, by item or, where there are more items than parts, by the part
// in which a split item begins: the grid is min(items, parts) x query rows of an item whatever the batch.
//
// What bounds it is a chain of memory round trips, merge_info -> (partial lse, partial rows) -> store, how often the middle
// is repeated, and how many blocks an SM can hold: the decode kernel of the next call is placed, and sets itself up, when
// the last of these blocks has started.  So a warp is kept to few registers, and takes
//   a row, up to four partials at a time, where there are many rows (more than eight per SM);
//   a quarter of a row, eight at a time, where there are few rows, and those of many partials;
//   half or a quarter of a row of FP32 partials (the kernel for few rows);
//   a quarter of a row and every fourth partial, the block's four warps adding up in shared memory, where a row has sixteen
//   partials or more on average: one sequence of 20000 keys (74 partials, nine batches one behind the other took 8-14 us)
//   22.0 -> 18.8 us, with 16 rows 17.7 -> 12.9; of 2531 keys 13.3 -> 12.6; of 6000 17.0 -> 15.1.
// Against a whole row per warp in 126 registers, eight partials at a time, and a warp for every row that an item has room
// for (the whole call): one sequence of 2531 keys 14.3 -> 13.2 us, of 60000 39.4 -> 35.1, of 3000 with 16 rows 12.4 -> 9.9;
// 192 sequences of 1-512 keys 45.4 -> 44.2; 32 of 1-8 K with 16 rows 37.5 -> 36.4; 96 of 2048 73.1 -> 71.7 cool.
// (One block per SM that walks over the rows and fits beside a decode CTA lets the next call's decode kernel in at once, but
// takes 10 us where these take 4: 32 x 4096 keys 55.8 -> 61.5.)
template <bool kFloat, int kCols, int kSplitWarps>
__global__ void __launch_bounds__(128, kCols == 16 ? 7 : kCols == 8 ? 8 : 5) combine_kernel(const __grid_constant__ DecodeParams prm) {
  // A decode kernel that follows on the stream may set itself up beside this kernel (it writes nothing this kernel
  // reads before its own wait for this kernel's completion).
  asm volatile("griddepcontrol.launch_dependents;");
  constexpr int kUnits = 16 / kCols;                       // warps per row
  constexpr int kFast = 4, kBatch = kCols == 16 || (kFloat && kCols == 8) ? 4 : 8;
  constexpr int kWords = kFloat ? kCols : kCols / 2;       // 32-bit words of a partial per lane
  const int lane = threadIdx.x & 31;
  const int sw = kSplitWarps == 1 ? 0 : threadIdx.x >> 5;  // takes the partials sw, sw + kSplitWarps, ...
  const int unit = kSplitWarps == 1 ? blockIdx.x * 4 + (threadIdx.x >> 5) : blockIdx.x;
  const int row = unit / kUnits, group = row / merge_rows(prm);
  const int rr = row - group * merge_rows(prm);            // row within the item
  const int col = (unit - row * kUnits) * (kDv / kUnits) + lane * kCols;
  asm volatile("griddepcontrol.wait;" ::: "memory");   // launched early (programmatic dependent launch): the partials must be complete
  if (group >= merge_groups(prm)) return;
  const int4 info = prm.merge_info[group];
  // (a decode kernel that gave up has perhaps not written it: what it names then need not exist)
  if (*prm.status != kStatusOk || info.z < 2) return;
  const int nsplit = (info.z - sw + kSplitWarps - 1) / kSplitWarps;      // of this warp
  const int b = prm.nrb == 1 ? info.x : info.x / prm.nrb;
  const int rin = (info.x - b * prm.nrb) * prm.item_rows + rr;                          // row within the sequence
  if (rin >= prm.R) return;

  auto part_row = [&](int s) { return static_cast<size_t>(Plan::slot_of_split(info.y, sw + kSplitWarps * s)) * prm.item_rows + rr; };
  struct Piece { uint32_t w[kWords], scale; };
  auto fetch = [&](int s) {
    const size_t prow = part_row(s);
    Piece x;
    const uint32_t* src = kFloat ? reinterpret_cast<const uint32_t*>(prm.part_o + prow * kDv + col) : reinterpret_cast<const uint32_t*>(partial_halves(prm) + prow * kDv + col);
    if constexpr (kWords == 2) {
      *reinterpret_cast<uint2*>(x.w) = *reinterpret_cast<const uint2*>(src);
    } else {
#pragma unroll
      for (int i = 0; i < kWords / 4; ++i) *reinterpret_cast<uint4*>(x.w + 4 * i) = reinterpret_cast<const uint4*>(src)[i];
    }
    if (!kFloat) x.scale = partial_scales(prm)[prow * 16 + col / 32];
    return x;
  };
  float acc[kCols], tot = 0.f;
#pragma unroll
  for (int i = 0; i < kCols; ++i) acc[i] = 0.f;
  auto accumulate = [&](float w, const Piece& x) {
    tot += w;
    const float ws = kFloat ? w : w * partial_unscale(x.scale);
#pragma unroll
    for (int i = 0; i < kWords; ++i) {
      if (kFloat) {
        acc[i] += ws * __uint_as_float(x.w[i]);
      } else {
        const float2 v = unpack_f16x2(x.w[i]);
        acc[2 * i % kCols] += ws * v.x;
        acc[(2 * i + 1) % kCols] += ws * v.y;
      }
    }
  };
  // the lse of 32 splits, one per lane, and the partials of a batch are on their way together
  float ls = lane < nsplit ? prm.part_lse[part_row(lane)] : -INFINITY;
  Piece x[kBatch];
  if (nsplit <= kFast) {
#pragma unroll
    for (int k = 0; k < kFast; ++k)
      if (k < nsplit) x[k] = fetch(k);
  } else {
#pragma unroll
    for (int k = 0; k < kBatch; ++k) x[k] = fetch(min(k, nsplit - 1));
  }
  float mx = ls;
  for (int s = lane + 32; s < nsplit; s += 32) mx = fmaxf(mx, prm.part_lse[part_row(s)]);
#pragma unroll
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (mx != -INFINITY) {                                   // else no split saw a visible key for this row: zeros
    ls = expf(ls - mx);                                    // 0 for a split that saw nothing
    if (nsplit <= kFast) {
#pragma unroll
      for (int k = 0; k < kFast; ++k)
        if (k < nsplit) accumulate(__shfl_sync(0xffffffffu, ls, k), x[k]);
    } else {
#pragma unroll 1
      for (int s0 = 0;;) {
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
          const float w = __shfl_sync(0xffffffffu, ls, (s0 + k) & 31);
          if (s0 + k < nsplit) accumulate(w, x[k]);
        }
        s0 += kBatch;
        if (s0 >= nsplit) break;
#pragma unroll
        for (int k = 0; k < kBatch; ++k) x[k] = fetch(min(s0 + k, nsplit - 1));
        if ((s0 & 31) == 0) ls = s0 + lane < nsplit ? expf(prm.part_lse[part_row(s0 + lane)] - mx) : 0.f;
      }
    }
  }
  if constexpr (kSplitWarps > 1) {
    static_assert(kCols == 4, "a lane's columns travel as one float4");
    __shared__ float4 s_acc[kSplitWarps][32];
    __shared__ float2 s_lse[kSplitWarps];
    s_acc[sw][lane] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    if (lane == 0) s_lse[sw] = make_float2(mx, tot);
    __syncthreads();
    if (sw != 0) return;
#pragma unroll
    for (int k = 1; k < kSplitWarps; ++k) mx = fmaxf(mx, s_lse[k].x);
    acc[0] = acc[1] = acc[2] = acc[3] = tot = 0.f;
    if (mx != -INFINITY) {
#pragma unroll
      for (int k = 0; k < kSplitWarps; ++k) {
        const float w = expf(s_lse[k].x - mx);
        const float4 v = s_acc[k][lane];
        tot += w * s_lse[k].y;
        acc[0] += w * v.x; acc[1] += w * v.y; acc[2] += w * v.z; acc[3] += w * v.w;
      }
    }
  }
  const float inv = tot > 0.f ? 1.f / tot : 0.f;
  uint32_t pk[kCols / 2];
#pragma unroll
  for (int i = 0; i < kCols / 2; ++i) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(acc[2 * i] * inv, acc[2 * i + 1] * inv);
    pk[i] = *reinterpret_cast<const uint32_t*>(&v);
  }
  __nv_bfloat16* dst = prm.out + (static_cast<size_t>(b) * prm.R + rin) * kDv + col;
  if constexpr (kCols == 4) {
    *reinterpret_cast<uint2*>(dst) = make_uint2(pk[0], pk[1]);
  } else {
#pragma unroll
    for (int i = 0; i < kCols / 8; ++i) reinterpret_cast<uint4*>(dst)[i] = make_uint4(pk[4 * i], pk[4 * i + 1], pk[4 * i + 2], pk[4 * i + 3]);
  }
  if (lane == 0 && col == 0) prm.lse[static_cast<size_t>(b) * prm.R + rin] = tot > 0.f ? mx + logf(tot) : -INFINITY;
}

cudaError_t launch_plan(const DecodeParams& prm, int* prefix_out, cudaStream_t stream) {
  plan_kernel<<<1, 1024, 0, stream>>>(prm.seqlens, prm.nrb, prm.n_items, prm.tile_keys, prm.ovh, prefix_out, prm.status);
  return cudaGetLastError();
}

cudaError_t launch_combine(const DecodeParams& prm, cudaStream_t stream) {
  const bool fp32 = prm.item_rows < kRowBlock;
  const int rows = merge_groups(prm) * merge_rows(prm);
  const bool few = rows <= 8 * prm.sms;
  const int units = rows * (few ? 4 : fp32 ? 2 : 1);
  const bool many = few && prm.P >= 16 * merge_groups(prm);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(many ? units : (units + 3) / 4);
  cfg.blockDim = dim3(128);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (many) return cudaLaunchKernelEx(&cfg, fp32 ? combine_kernel<true, 4, 4> : combine_kernel<false, 4, 4>, prm);
  if (few) return cudaLaunchKernelEx(&cfg, fp32 ? combine_kernel<true, 4, 1> : combine_kernel<false, 4, 1>, prm);
  return cudaLaunchKernelEx(&cfg, fp32 ? combine_kernel<true, 8, 1> : combine_kernel<false, 16, 1>, prm);
}

}  // namespace amla
