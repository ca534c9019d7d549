// Arithmetic-pipe throughput of the GPU, measured the way the roofline denominators of the
// benchmark need them: every thread runs CHAINS independent fused multiply-add chains (enough
// independent work per warp to hide the pipe latency) for `iters` rounds, and the launch's
// CUDA-event time gives the FMA rate.  FP64 (DFMA), binary32 (FFMA) and the 32 x 32 + 64-bit integer
// multiply-add of the fixed-point contractions.  The chains' values stay finite and are written
// out, so no work is removed by the compiler.
#include <cuda_runtime.h>

namespace {
constexpr int CHAINS = 8;

template <typename T>
__global__ void __launch_bounds__(256) k_fma_chains(T* sink, int iters, T a, T b) {
  T x[CHAINS];
#pragma unroll
  for (int c = 0; c < CHAINS; ++c) x[c] = (T)(threadIdx.x + c) * (T)1e-3;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int c = 0; c < CHAINS; ++c) x[c] = fma(x[c], a, b);
  }
  T s = 0;
#pragma unroll
  for (int c = 0; c < CHAINS; ++c) s += x[c];
  sink[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

// Accumulations of one product, as a contraction's; asm, so that they are not folded into one.
__global__ void __launch_bounds__(256) k_mad_chains(long long* sink, int iters, int b) {
  long long x[CHAINS];
  const int a = (int)threadIdx.x * b;
#pragma unroll
  for (int c = 0; c < CHAINS; ++c) x[c] = threadIdx.x + c;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int c = 0; c < CHAINS; ++c)
      asm volatile("mad.wide.s32 %0, %1, %2, %0;" : "+l"(x[c]) : "r"(a), "r"(b));
  }
  long long s = 0;
#pragma unroll
  for (int c = 0; c < CHAINS; ++c) s += x[c];
  sink[blockIdx.x * blockDim.x + threadIdx.x] = s;
}
}  // namespace

extern "C" {

// Launch `blocks` x 256 threads, each with 8 chains of `iters` FMA (2 flops each) in binary32 (kind
// 0) or FP64 (1), or of integer multiply-adds (2); `sink` must hold blocks * 256 elements of that
// type, 4 or 8 bytes (device memory).  Returns the cudaError_t of the launch.  The multiplier 0.999
// and addend 1e-3 keep each chain bounded.
int peaks_fma_launch(int kind, void* sink, int blocks, int iters, void* stream) {
  if (blocks < 1 || iters < 1 || !sink) return (int)cudaErrorInvalidValue;
  cudaStream_t s = (cudaStream_t)stream;
  if (kind == 2)
    k_mad_chains<<<blocks, 256, 0, s>>>((long long*)sink, iters, 12345);
  else if (kind == 1)
    k_fma_chains<double><<<blocks, 256, 0, s>>>((double*)sink, iters, 0.999, 1e-3);
  else
    k_fma_chains<float><<<blocks, 256, 0, s>>>((float*)sink, iters, 0.999f, 1e-3f);
  return (int)cudaGetLastError();
}

// Flops of one launch: blocks x 256 threads x 8 chains x iters x 2 (integers: twice the multiply-adds).
double peaks_fma_flops(int blocks, int iters) {
  return (double)blocks * 256.0 * CHAINS * (double)iters * 2.0;
}

}  // extern "C"
