// Test aid: a producer of sequence lengths that lets the kernel behind it on the stream start at once (programmatic
// dependent launch) and writes the lengths a while later.  Whoever reads them before griddepcontrol.wait finds what the
// buffer held before.
#include <cuda_runtime.h>

__global__ void late_lengths_kernel(const int* src, int* dst, int n, unsigned long long delay_ns) {
  asm volatile("griddepcontrol.launch_dependents;");
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
  for (int i = 0; i < 1 << 16; ++i) {                   // bounded whatever the timer does
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    if (t - t0 >= delay_ns) break;
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

extern "C" int late_lengths(const int* src, int* dst, int n, unsigned long long delay_ns, void* stream) {
  if (!src || !dst || n <= 0 || delay_ns > 1000000ull) return -1;
  late_lengths_kernel<<<1, 256, 0, static_cast<cudaStream_t>(stream)>>>(src, dst, n, delay_ns);
  return cudaGetLastError() == cudaSuccess ? 0 : -4;
}
