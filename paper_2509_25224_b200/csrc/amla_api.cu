// C-ABI entry points of libamla: argument validation, workspace carving and the three launches
// (schedule prefix, decode, combine) on the caller's stream.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <new>

#include "../../include/amla.h"
#include "amla_common.cuh"

namespace amla {
cudaError_t launch_plan(const DecodeParams& prm, int* prefix_out, cudaStream_t stream);
cudaError_t launch_combine(const DecodeParams& prm, cudaStream_t stream);
cudaError_t launch_decode_simt(const DecodeParams& prm, cudaStream_t stream);
// Returns cudaSuccess, or an error; sets *unsupported when the device cannot run the kernel.
cudaError_t launch_decode_pair(const DecodeParams& prm, cudaStream_t stream, int* unsupported);
cudaError_t launch_decode_few(const DecodeParams& prm, cudaStream_t stream, int* unsupported);
cudaError_t launch_decode_quad(const DecodeParams& prm, cudaStream_t stream, int* unsupported);
cudaError_t launch_wait_selftest(int* status, unsigned long long limit_ns, cudaStream_t stream);
cudaError_t launch_widen_pages(const uint8_t* kv8, const int32_t* block_table, const int32_t* seqlens, int B, int num_blocks,
                               int max_blocks_per_seq, __nv_bfloat16* scratch, int32_t* table_out, cudaStream_t stream);
int decode_pair_parts(int sm_count);
int decode_quad_parts(int device, int sm_count);

namespace {

constexpr size_t kAlign = 256;
constexpr int kMaxRows = 1024;   // Sq * H

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

struct Layout {
  size_t status_off, merge_off, prefix_off, part_lse_off, part_o_off, total;
};

Layout make_layout(int n_items, int max_parts) {
  Layout l;
  l.status_off = 0;
  l.merge_off = kAlign;
  l.prefix_off = l.merge_off + align_up(sizeof(int4) * static_cast<size_t>(max_parts));
  l.part_lse_off = l.prefix_off + align_up(sizeof(int) * (static_cast<size_t>(n_items) + 1));
  l.part_o_off = l.part_lse_off + align_up(sizeof(float) * 2 * static_cast<size_t>(max_parts) * kRowBlock);
  l.total = l.part_o_off + sizeof(float) * 2 * static_cast<size_t>(max_parts) * kRowBlock * kDv;
  return l;
}

int check_shape(int B, int Sq, int H, int max_blocks_per_seq) {
  if (B <= 0 || Sq <= 0 || H <= 0 || max_blocks_per_seq <= 0) return AMLA_ERR_INVALID_ARG;
  if (Sq > 8 || H > 128 || Sq * H > kMaxRows) return AMLA_ERR_UNSUPPORTED;
  if (static_cast<long long>(max_blocks_per_seq) * kPage > (1ll << 30)) return AMLA_ERR_UNSUPPORTED;
  if (static_cast<long long>(B) * ((Sq * H + kRowBlock - 1) / kRowBlock) > (1ll << 24)) return AMLA_ERR_UNSUPPORTED;
  return AMLA_OK;
}

// SM count and compute capability per device, queried once (the attributes never change).
constexpr int kMaxDevices = 64;
struct DeviceInfo { std::atomic<int> ready{0}; int sms = 0; int cc_major = 0; };
DeviceInfo g_devices[kMaxDevices];

int sm_count_of(int device, int* sms, int* cc_major) {
  if (device < 0 || device >= kMaxDevices) return AMLA_ERR_INVALID_ARG;
  DeviceInfo& d = g_devices[device];
  if (!d.ready.load(std::memory_order_acquire)) {
    int s = 0, c = 0;
    if (cudaDeviceGetAttribute(&s, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaDeviceGetAttribute(&c, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess) {
      cudaGetLastError();
      return AMLA_ERR_CUDA;
    }
    d.sms = s; d.cc_major = c;
    d.ready.store(1, std::memory_order_release);
  }
  *sms = d.sms;
  *cc_major = d.cc_major;
  return AMLA_OK;
}

thread_local int g_last_launches = 0, g_last_item_rows = 0;
#ifdef AMLA_TRACE
thread_local unsigned long long* g_trace = nullptr;
#endif

// Optional per-kernel timing (measurement aid): four events bracketing the three launches.
thread_local bool g_profile = false;
thread_local cudaEvent_t g_ev[4] = {nullptr, nullptr, nullptr, nullptr};
thread_local bool g_ev_valid = false;

void profile_mark(int i, cudaStream_t stream) {
  if (g_profile && g_ev[i]) { cudaEventRecord(g_ev[i], stream); if (i == 3) g_ev_valid = true; }
}

}  // namespace

// Sequences with more than 128 query rows: blocks of 256 rows on four SMs, or independent blocks of 128 rows on two?  The
// 256-row kernel reads the cache once for 256 rows, but a call of it takes longer to start and to finish, and so does every
// further item that a part begins.  What either takes was measured over 1-200 sequences of 64-60000 keys and 2-8 tokens:
//   256 rows: 21.5 us + 2.08 us per 128-key tile of a part + 11 us per item of a part beyond the first
//   128 rows: 13 us + 1.41 us per page of a part + 6 us per item of a part
// (The figures are from before units of the 128-row kernel ran into one another and the next tile's K came by way of L2.  70 shapes
// in short bursts since: 21.0 + 1.99 + 10.4 and 13.5 + 1.11 + 5.8.  Which calls take which kernel has not been gone over with that:
// long calls run at the power limit, where reading the cache once counts for more than a burst shows.)
// e.g. (two tokens, 128 heads) 1 x 3000 keys 22.0 against 15.7 us, 32 x 256 23.4 / 21.8, 32 x 2000 49 / 57, 1 x 60000 47.9 / 48.8.
// Lengths are not known here: the block table's width bounds them.
static bool blocks_of_256(const DecodeParams& prm, int pair_parts, int quad_parts) {
  const double pages = prm.max_blocks_per_seq, tiles = (prm.max_blocks_per_seq + 1) / 2;
  const double items1 = static_cast<double>(prm.B) * ((prm.R + kRowBlock - 1) / kRowBlock) / pair_parts;
  const double items2 = static_cast<double>(prm.B) * ((prm.R + 2 * kRowBlock - 1) / (2 * kRowBlock)) / quad_parts;
  return 21.5 + 2.08 * items2 * tiles + 11. * std::max(items2 - 1., 0.) < 13. + 1.41 * items1 * pages + 6. * items1;
}

// Chooses the kernel for the shape and fills the schedule fields of prm (rows per item, keys per tile, parts):
//   up to 32 query rows of a bf16 cache      the kernel for few rows
//   more than 128 rows of a bf16 cache       the 256-row kernel (four-CTA clusters, pair MMAs) where it is the faster one
//   everything else                          the 128-row kernel
// AMLA_FLAG_KERNEL_ROWS128 asks for the 128-row kernel whatever the shape.
int configure_schedule(DecodeParams& prm, int device, int sms, int flags) {
  prm.sms = sms;
  const bool simt = (flags & AMLA_FLAG_KERNEL_SIMT) != 0;
  bool quad = !simt && !(flags & AMLA_FLAG_KERNEL_ROWS128) && prm.R > kRowBlock && prm.kv8 == nullptr;
  int quad_parts = 0;
  if (quad) {
    quad_parts = decode_quad_parts(device, sms);
    if (quad_parts <= 0 || !blocks_of_256(prm, decode_pair_parts(sms), quad_parts)) quad = false;   // (0: four-CTA clusters cannot be placed on this device)
  }
  // A single sequence of at most four pages is one score tile of the 128-row kernel, and the kernel for few rows would take
  // it a page at a time: 256 keys, 16 rows 8.4 us against 8.6, 32 rows 8.8 against 10.0 (64 keys 8.3 against 8.2).
  const bool one_tile = prm.B == 1 && prm.max_blocks_per_seq <= 4;
  const bool few = !simt && !(flags & AMLA_FLAG_KERNEL_ROWS128) && prm.R <= kFewRows && prm.kv8 == nullptr && !one_tile;
  prm.item_rows = quad ? 2 * kRowBlock : few ? kFewRows : kRowBlock;
  prm.tile_keys = quad ? 2 * kPage : kPage;
  prm.ovh = quad ? kQuadOverheadTiles : few ? kFewOverheadTiles : kUnitOverheadTiles;
  // (tau = 0 asks for Algorithm 2 to the letter: its parts stay as fine as the schedule's tiles, so that a short sequence
  // is summed in blocks of 64 keys)
  prm.min_share = simt || (flags & AMLA_LAZY_MASK) == 0 ? 1 : kMinPartKeys / prm.tile_keys;
  prm.nrb = (prm.R + prm.item_rows - 1) / prm.item_rows;
  prm.n_items = prm.B * prm.nrb;
  prm.P = simt || few ? sms : quad ? quad_parts : decode_pair_parts(sms);
  // No more parts than the longest schedule that the block table's width allows can fill.  A schedule of one score tile at
  // most is one part: nothing is split and no combine kernel runs.
  const long long tiles = (static_cast<long long>(prm.max_blocks_per_seq) * kPage + prm.tile_keys - 1) / prm.tile_keys;
  const long long longest = prm.n_items * tiles + (prm.n_items - 1ll) * prm.ovh;
  if (!simt) {
    if (longest * prm.tile_keys <= 256) prm.P = 1;
    else prm.P = static_cast<int>(std::min<long long>(prm.P, (longest + prm.min_share - 1) / prm.min_share));
  }
  // (a plan made in the decode kernel may begin as a guess: any lengths that the table has room for must add up)
  prm.fused_plan = (!simt && prm.n_items <= kFusedPlanMaxItems && longest <= 0x7fffffff) ? 1 : 0;
  return AMLA_OK;
}

// The launches of one decode call (schedule kernel for large batches, decode, combine) on `stream`.
int launch_decode_call(const DecodeParams& prm, int* prefix, cudaStream_t stream, int* launches, void (*mark)(int, cudaStream_t)) {
  const bool simt = (prm.flags & AMLA_FLAG_KERNEL_SIMT) != 0;
  g_last_item_rows = prm.item_rows;
  if (mark) mark(0, stream);
  if (!prm.fused_plan) {
    if (launch_plan(prm, prefix, stream) != cudaSuccess) { cudaGetLastError(); return AMLA_ERR_CUDA; }
    ++*launches;
  }
  if (mark) mark(1, stream);
  if (simt) {
    if (launch_decode_simt(prm, stream) != cudaSuccess) { cudaGetLastError(); return AMLA_ERR_CUDA; }
  } else {
    int unsupported = 0;
    const cudaError_t err = prm.item_rows > kRowBlock   ? launch_decode_quad(prm, stream, &unsupported)
                            : prm.item_rows < kRowBlock ? launch_decode_few(prm, stream, &unsupported)
                                                        : launch_decode_pair(prm, stream, &unsupported);
    if (err != cudaSuccess) {
      cudaGetLastError();
      return unsupported ? AMLA_ERR_UNSUPPORTED : AMLA_ERR_CUDA;
    }
  }
  ++*launches;
  if (mark) mark(2, stream);
  if (prm.P > 1) {
    if (launch_combine(prm, stream) != cudaSuccess) { cudaGetLastError(); return AMLA_ERR_CUDA; }
    ++*launches;
  }
  if (mark) mark(3, stream);
  return AMLA_OK;
}

}  // namespace amla

using namespace amla;

extern "C" const char* amla_status_string(int status) {
  switch (status) {
    case AMLA_OK: return "ok";
    case AMLA_ERR_INVALID_ARG: return "invalid argument";
    case AMLA_ERR_UNSUPPORTED: return "unsupported shape or device";
    case AMLA_ERR_WORKSPACE: return "workspace too small";
    case AMLA_ERR_CUDA: return "CUDA call failed";
    case AMLA_ERR_DEVICE_TIMEOUT: return "device-side wait timed out";
    case AMLA_ERR_STATIC_LIMIT: return "problem or device exceeds the built-in scratch of amla_mla_decode_static";
    default: return "unknown status";
  }
}

extern "C" int amla_mla_decode_workspace_size(int B, int Sq, int H, int max_blocks_per_seq, int device,
                                              size_t* bytes_out) {
  if (!bytes_out) return AMLA_ERR_INVALID_ARG;
  int rc = check_shape(B, Sq, H, max_blocks_per_seq);
  if (rc != AMLA_OK) return rc;
  int sms = 0, cc = 0;
  rc = sm_count_of(device, &sms, &cc);
  if (rc != AMLA_OK) return rc;
  const int nrb = (Sq * H + kRowBlock - 1) / kRowBlock;
  *bytes_out = make_layout(B * nrb, sms).total;
  return AMLA_OK;
}

namespace {

// What can be said about a call's arguments without a device.
int check_arguments(const void* q, const void* cache, const int32_t* block_table, const int32_t* seqlens, float softmax_scale, int B, int Sq, int H,
                    int num_blocks, int max_blocks_per_seq, const void* out, const float* lse, const void* workspace, int flags) {
  if (!q || !cache || !block_table || !seqlens || !out || !lse || !workspace) return AMLA_ERR_INVALID_ARG;
  if (num_blocks <= 0 || !(softmax_scale == softmax_scale)) return AMLA_ERR_INVALID_ARG;
  const int rc = check_shape(B, Sq, H, max_blocks_per_seq);
  if (rc != AMLA_OK) return rc;
  if ((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(cache) | reinterpret_cast<uintptr_t>(out)) & 15) return AMLA_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(block_table) | reinterpret_cast<uintptr_t>(seqlens) | reinterpret_cast<uintptr_t>(lse)) & 3)
    return AMLA_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(workspace) & (kAlign - 1)) return AMLA_ERR_INVALID_ARG;
  if ((flags & AMLA_RESCALE_MASK) == 3) return AMLA_ERR_INVALID_ARG;
  return AMLA_OK;
}

// The decode call on a bf16 cache (kv_cache) or an E4M3 cache (kv8).  out_scale multiplies the normalised output (1 unless the cache was widened from
// FP8 with a dequantisation scale); launches are added to g_last_launches.
int decode_impl(const void* q, const void* kv_cache, const uint8_t* kv8, const int32_t* block_table, const int32_t* seqlens,
                float softmax_scale, float out_scale, int B, int Sq, int H, int num_blocks, int max_blocks_per_seq,
                void* out, float* lse, void* workspace, size_t workspace_bytes, void* cuda_stream, int flags) {
  int rc = check_arguments(q, kv8 ? static_cast<const void*>(kv8) : kv_cache, block_table, seqlens, softmax_scale, B, Sq, H, num_blocks, max_blocks_per_seq,
                           out, lse, workspace, flags);
  if (rc != AMLA_OK) return rc;

  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess) { cudaGetLastError(); return AMLA_ERR_CUDA; }
  int sms = 0, cc = 0;
  rc = sm_count_of(device, &sms, &cc);
  if (rc != AMLA_OK) return rc;
  if (cc != 10) return AMLA_ERR_UNSUPPORTED;

  // the layout is sized for 128-row items (the larger item count) whichever kernel runs
  const Layout lay = make_layout(B * ((Sq * H + kRowBlock - 1) / kRowBlock), sms);
  if (workspace_bytes < lay.total) return AMLA_ERR_WORKSPACE;

  char* ws = static_cast<char*>(workspace);
  DecodeParams prm;
  std::memset(&prm, 0, sizeof(prm));
  prm.q = static_cast<const __nv_bfloat16*>(q);
  prm.kv = static_cast<const __nv_bfloat16*>(kv_cache);
  prm.kv8 = kv8;
  prm.block_table = block_table;
  prm.seqlens = seqlens;
  prm.out = static_cast<__nv_bfloat16*>(out);
  prm.lse = lse;
  prm.status = reinterpret_cast<int*>(ws + lay.status_off);
  int* prefix = reinterpret_cast<int*>(ws + lay.prefix_off);
  prm.prefix = prefix;
  prm.merge_info = reinterpret_cast<int4*>(ws + lay.merge_off);
  prm.part_lse = reinterpret_cast<float*>(ws + lay.part_lse_off);
  prm.part_o = reinterpret_cast<float*>(ws + lay.part_o_off);
  prm.scale_log2 = softmax_scale * kLog2e;
  prm.out_scale = out_scale;
  prm.B = B; prm.Sq = Sq; prm.H = H;
  prm.R = Sq * H;
  prm.num_blocks = num_blocks;
  prm.max_blocks_per_seq = max_blocks_per_seq;
  prm.flags = flags;
#ifdef AMLA_TRACE
  prm.trace = g_trace;
#endif
  prm.tau = static_cast<float>((flags & AMLA_LAZY_MASK) >> AMLA_LAZY_SHIFT);
  rc = configure_schedule(prm, device, sms, flags);
  if (rc != AMLA_OK) return rc;
  return launch_decode_call(prm, prefix, static_cast<cudaStream_t>(cuda_stream), &g_last_launches, profile_mark);
}

// Are the pages of an E4M3 cache widened into a bf16 copy first, and the bf16 kernels run on that, or does the 128-row kernel
// widen them on their way in?  On their way in they are widened once more for every 128 query rows, and for K and for V; the
// copy costs its writing and reading once, and more than 128 rows then are blocks of 256.  Measured (on the way in / copy
// first, 128 heads, us): eight tokens 32 x 4096 keys 387 / 325, 16 x 16384 744 / 561, 64 x 1000 227 / 182; six tokens 275 / 253,
// 551 / 452; but five and less differ by little or the other way (32 x 4096 220, 1 x 4096 20.6 / 21.0, two tokens 32 x 4096
// 98 / 130), and so do small calls (1 x 100, six tokens 12.1 / 13.6; 20 x 375-3000 79.7 / 81.0).  Lengths are not known here: the
// table's width stands for them, unless the cache could not fill half of such a table (100 sequences of 300 keys, six tokens, a
// table of 512 pages: 141 / 184).  (The scalar bring-up kernel reads bf16 only.)
bool widen_first(int B, int rows, int num_blocks, int max_blocks_per_seq, int flags) {
  if (flags & AMLA_FLAG_KERNEL_SIMT) return true;
  const long long row_blocks = (rows + kRowBlock - 1) / kRowBlock, slots = static_cast<long long>(B) * max_blocks_per_seq;
  return !(flags & AMLA_FLAG_KERNEL_ROWS128) && row_blocks > 5 && row_blocks * slots >= 8192 && slots <= 2ll * num_blocks;
}

// Bytes of the FP8 path's extra scratch behind the ordinary workspace: the new block table and the widened pages.
size_t fp8_table_bytes(int B, int max_blocks_per_seq) { return align_up(sizeof(int32_t) * static_cast<size_t>(B) * max_blocks_per_seq); }
size_t fp8_pages_bytes(int B, int max_blocks_per_seq) { return static_cast<size_t>(B) * max_blocks_per_seq * kPage * kDqk * sizeof(__nv_bfloat16); }

}  // namespace

extern "C" int amla_mla_decode_ex(const void* q, const void* kv_cache, const int32_t* block_table,
                                  const int32_t* seqlens, float softmax_scale, int B, int Sq, int H,
                                  int num_blocks, int max_blocks_per_seq, void* out, float* lse,
                                  void* workspace, size_t workspace_bytes, void* cuda_stream, int flags) {
  g_last_launches = 0;
  return decode_impl(q, kv_cache, nullptr, block_table, seqlens, softmax_scale, 1.f, B, Sq, H, num_blocks, max_blocks_per_seq, out, lse,
                     workspace, workspace_bytes, cuda_stream, flags);
}

extern "C" int amla_mla_decode_fp8_workspace_size(int B, int Sq, int H, int max_blocks_per_seq, int device, size_t* bytes_out) {
  size_t base = 0;
  const int rc = amla_mla_decode_workspace_size(B, Sq, H, max_blocks_per_seq, device, &base);
  if (rc != AMLA_OK) return rc;
  *bytes_out = align_up(base) + fp8_table_bytes(B, max_blocks_per_seq) + fp8_pages_bytes(B, max_blocks_per_seq);
  return AMLA_OK;
}

extern "C" int amla_mla_decode_fp8(const void* q, const void* kv_cache_e4m3, float kv_scale, const int32_t* block_table,
                                   const int32_t* seqlens, float softmax_scale, int B, int Sq, int H, int num_blocks,
                                   int max_blocks_per_seq, void* out, float* lse, void* workspace, size_t workspace_bytes,
                                   void* cuda_stream, int flags) {
  g_last_launches = 0;
  // (all of it here: the widening kernel is launched ahead of decode_impl)
  int rc = check_arguments(q, kv_cache_e4m3, block_table, seqlens, softmax_scale, B, Sq, H, num_blocks, max_blocks_per_seq, out, lse, workspace, flags);
  if (rc != AMLA_OK) return rc;
  if (!(kv_scale == kv_scale) || !(softmax_scale * kv_scale == softmax_scale * kv_scale)) return AMLA_ERR_INVALID_ARG;
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess) { cudaGetLastError(); return AMLA_ERR_CUDA; }
  size_t base = 0;
  rc = amla_mla_decode_workspace_size(B, Sq, H, max_blocks_per_seq, device, &base);
  if (rc != AMLA_OK) return rc;
  base = align_up(base);
  const size_t tbytes = fp8_table_bytes(B, max_blocks_per_seq), pbytes = fp8_pages_bytes(B, max_blocks_per_seq);
  if (workspace_bytes < base + tbytes + pbytes) return AMLA_ERR_WORKSPACE;
  if (static_cast<long long>(B) * max_blocks_per_seq > (1ll << 30)) return AMLA_ERR_UNSUPPORTED;
  // logits: scale * q . (k8 * kv_scale); output: sum p * (v8 * kv_scale)
  if (!widen_first(B, Sq * H, num_blocks, max_blocks_per_seq, flags))
    return decode_impl(q, nullptr, static_cast<const uint8_t*>(kv_cache_e4m3), block_table, seqlens, softmax_scale * kv_scale, kv_scale, B, Sq, H,
                       num_blocks, max_blocks_per_seq, out, lse, workspace, base, cuda_stream, flags);
  char* ws = static_cast<char*>(workspace);
  int32_t* table2 = reinterpret_cast<int32_t*>(ws + base);
  __nv_bfloat16* pages = reinterpret_cast<__nv_bfloat16*>(ws + base + tbytes);
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  if (launch_widen_pages(static_cast<const uint8_t*>(kv_cache_e4m3), block_table, seqlens, B, num_blocks, max_blocks_per_seq,
                         pages, table2, stream) != cudaSuccess) {
    cudaGetLastError();
    return AMLA_ERR_CUDA;
  }
  ++g_last_launches;
  return decode_impl(q, pages, nullptr, table2, seqlens, softmax_scale * kv_scale, kv_scale, B, Sq, H, B * max_blocks_per_seq,
                     max_blocks_per_seq, out, lse, workspace, base, cuda_stream, flags);
}

extern "C" int amla_mla_decode(const void* q, const void* kv_cache, const int32_t* block_table,
                               const int32_t* seqlens, float softmax_scale, int B, int Sq, int H,
                               int num_blocks, int max_blocks_per_seq, void* out, float* lse,
                               void* workspace, size_t workspace_bytes, void* cuda_stream) {
  return amla_mla_decode_ex(q, kv_cache, block_table, seqlens, softmax_scale, B, Sq, H, num_blocks,
                            max_blocks_per_seq, out, lse, workspace, workspace_bytes, cuda_stream,
                            AMLA_RESCALE_ALG2 | AMLA_LAZY(AMLA_DEFAULT_TAU));
}

extern "C" int amla_check_status(const void* workspace, void* cuda_stream) {
  if (!workspace) return AMLA_ERR_INVALID_ARG;
  int st = 0;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMemcpyAsync(&st, workspace, sizeof(int), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess) {
    cudaGetLastError();
    return AMLA_ERR_CUDA;
  }
  return st == kStatusOk ? AMLA_OK : AMLA_ERR_DEVICE_TIMEOUT;
}

extern "C" int amla_last_launch_count(void) { return g_last_launches; }
extern "C" int amla_last_item_rows(void) { return g_last_item_rows; }

extern "C" int amla_wait_selftest(void* workspace, unsigned long long limit_ns, void* cuda_stream) {
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 3)) return AMLA_ERR_INVALID_ARG;
  if (limit_ns == 0 || limit_ns > 100000000ull) return AMLA_ERR_INVALID_ARG;      // at most 0.1 s
  if (launch_wait_selftest(static_cast<int*>(workspace), limit_ns, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess) {
    cudaGetLastError();
    return AMLA_ERR_CUDA;
  }
  return AMLA_OK;
}

extern "C" int amla_validate_paging_host(const int32_t* block_table, const int32_t* seqlens, int B, int num_blocks,
                                         int max_blocks_per_seq, int* bad_seq, int* bad_block) {
  if (!block_table || !seqlens || B <= 0 || num_blocks <= 0 || max_blocks_per_seq <= 0) return AMLA_ERR_INVALID_ARG;
  for (int b = 0; b < B; ++b) {
    const long long n = seqlens[b];
    if (n < 0 || n > static_cast<long long>(max_blocks_per_seq) * kPage) {
      if (bad_seq) *bad_seq = b;
      if (bad_block) *bad_block = -1;
      return AMLA_ERR_INVALID_ARG;
    }
    const int used = static_cast<int>((n + kPage - 1) / kPage);
    for (int i = 0; i < used; ++i) {
      const int32_t pg = block_table[static_cast<size_t>(b) * max_blocks_per_seq + i];
      if (pg < 0 || pg >= num_blocks) {
        if (bad_seq) *bad_seq = b;
        if (bad_block) *bad_block = i;
        return AMLA_ERR_INVALID_ARG;
      }
    }
  }
  return AMLA_OK;
}

extern "C" int amla_profile_enable(int on) {
  if (on && !g_ev[0]) {
    for (int i = 0; i < 4; ++i) {
      if (cudaEventCreate(&g_ev[i]) != cudaSuccess) { cudaGetLastError(); g_ev[i] = nullptr; return AMLA_ERR_CUDA; }
    }
  }
  g_profile = on != 0;
  g_ev_valid = false;
  return AMLA_OK;
}

extern "C" int amla_profile_last_ms(float* ms3) {
  if (!ms3) return AMLA_ERR_INVALID_ARG;
  if (!g_ev_valid) return AMLA_ERR_INVALID_ARG;
  if (cudaEventSynchronize(g_ev[3]) != cudaSuccess) { cudaGetLastError(); return AMLA_ERR_CUDA; }
  for (int i = 0; i < 3; ++i) {
    if (cudaEventElapsedTime(&ms3[i], g_ev[i], g_ev[i + 1]) != cudaSuccess) { cudaGetLastError(); return AMLA_ERR_CUDA; }
  }
  return AMLA_OK;
}

extern "C" int amla_plan_host(const int32_t* seqlens, int B, int Sq, int H, int num_parts, int32_t* units,
                              int max_units) {
  if (!seqlens || !units || num_parts <= 0 || max_units < 0) return AMLA_ERR_INVALID_ARG;
  int rc = check_shape(B, Sq, H, 1);
  if (rc != AMLA_OK) return rc;
  const bool quad = Sq * H > kRowBlock, few = Sq * H <= kFewRows;
  const int item_rows = quad ? 2 * kRowBlock : few ? kFewRows : kRowBlock, tile_keys = quad ? 2 * kPage : kPage;
  const int ovh = quad ? kQuadOverheadTiles : few ? kFewOverheadTiles : kUnitOverheadTiles;
  const int nrb = (Sq * H + item_rows - 1) / item_rows;
  const int n_items = B * nrb;
  int* prefix = new (std::nothrow) int[n_items + 1];
  if (!prefix) return AMLA_ERR_WORKSPACE;
  int acc = 0;
  for (int it = 0; it < n_items; ++it) {
    prefix[it] = acc;
    acc += schedule_length(seqlens[it / nrb], it, tile_keys, ovh);
  }
  prefix[n_items] = acc;
  const Plan plan = Plan::make(prefix, n_items, num_parts, ovh, kMinPartKeys / tile_keys);
  int n_units = 0;
  bool overflow = false;
  if (acc > 0) {
    for (int p = 0; p < plan.P; ++p) {
      const int g0 = plan.part_start(p), g1 = plan.part_start(p + 1);
      int g = g0;
      while (g < g1) {
        const int it = plan.item_of_tile(g);
        const int a = plan.first_tile(it), e = prefix[it + 1];
        const int lo = g > a ? g : a, hi = e < g1 ? e : g1;
        g = e < g1 ? e : g1;
        if (hi <= lo) continue;
        const int t0 = lo - a, t1 = hi - a;
        int p_first, p_last;
        const int nsplit = plan.item_parts(it, &p_first, &p_last);
        if (n_units < max_units) {
          int32_t* u = units + 6 * n_units;
          u[0] = p; u[1] = it; u[2] = t0; u[3] = t1;
          u[4] = nsplit == 1 ? -1 : plan.slot_of(p, it, p_first);
          u[5] = nsplit;
        } else {
          overflow = true;
        }
        ++n_units;
      }
    }
  }
  delete[] prefix;
  return overflow ? AMLA_ERR_WORKSPACE : n_units;
}

#ifdef AMLA_TRACE
// Trace builds only (not part of the public header): device buffer of
// parts * kTraceEvents * kTraceTiles 64-bit stamps that later calls on this thread fill.
extern "C" int amla_debug_set_trace(void* device_buffer) {
  g_trace = static_cast<unsigned long long*>(device_buffer);
  return AMLA_OK;
}
#endif
