// The log-space L1 loss (Sec. 5) of an FP32 batch and its derivative in one
// pass, for callers that own the loss themselves:
//   mean |log(1 + max(g, 0)) - log(1 + y)| + 0.01 max(-g, 0).
// Written out in tensor operations it is ten launches forward and twelve
// backward, each of a few microseconds of device time behind as much or more
// of host time; here it is two launches (the second adds up the blocks' sums,
// in a fixed order), and a scaling of the derivative when the gradient comes
// back.  A training iteration of 50,000 queries through autograd: 370 us, with
// the tensor operations 636.
#include <cuda_runtime.h>

#include "nam_ctx.h"

namespace nam {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ double block_sum(double v) {
  __shared__ double s[kThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) t += s[w];
  return t;
}

// unit, copy (may be null, both or neither): d(mean)/dg, and g again.  Zeros, infinities and NaN as the tensor
// operations' derivatives have them: sign is 0 at 0 and NaN, no gradient through
// max(g, 0) at g <= 0.
__global__ void __launch_bounds__(kThreads) log_l1_kernel(const float* __restrict__ g, const float* __restrict__ y,
                                                          int64_t n, float inv_n, float* __restrict__ unit,
                                                          float* __restrict__ copy, double* __restrict__ partial) {
  float sum = 0.0f;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) {
    const float x = g[i];
    const float r = x <= 0.0f ? 0.0f : x, neg = -x <= 0.0f ? 0.0f : -x;  // (NaN stays NaN)
    const float d = log1pf(r) - log1pf(y[i]);
    sum += fabsf(d) + 0.01f * neg;
    if (unit) {
      const float s = d > 0.0f ? inv_n : d < 0.0f ? -inv_n : 0.0f;
      const float a = x <= 0.0f ? 0.0f : s / (r + 1.0f);
      unit[i] = -x <= 0.0f ? a : a - 0.01f * inv_n;
      copy[i] = x;
    }
  }
  const double t = block_sum(sum);
  if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kThreads) log_l1_mean_kernel(const double* __restrict__ partial, int blocks, int64_t n,
                                                               float* __restrict__ loss) {
  double v = 0.0;
  for (int i = threadIdx.x; i < blocks; i += kThreads) v += partial[i];
  v = block_sum(v);
  if (threadIdx.x == 0) *loss = (float)(v / (double)n);
}

}  // namespace
}  // namespace nam

// Internal to the Python package (autograd.log_l1_loss), on the current
// device: loss[0], unit[n] and copy[n] or null; work: n_work doubles, as many
// as there are blocks at most.
extern "C" nam_status nam_internal_log_l1(const float* g, const float* y, int64_t n, float* unit, float* copy,
                                          float* loss, double* work, int64_t n_work, void* stream) {
  using namespace nam;
  if (n_work < 1) return fail(NAM_ERR_INVALID_ARG, "log_l1: no workspace");
  if (n < 1) return fail(NAM_ERR_INVALID_ARG, "log_l1: no values");
  const int64_t want = (n + 4 * kThreads - 1) / (4 * kThreads);
  const int64_t cap = n_work < 65535 ? n_work : 65535;
  const int blocks = (int)(want < cap ? want : cap);
  cudaStream_t s = (cudaStream_t)stream;
  log_l1_kernel<<<blocks, kThreads, 0, s>>>(g, y, n, 1.0f / (float)n, unit, copy, work);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) {
    log_l1_mean_kernel<<<1, kThreads, 0, s>>>(work, blocks, n, loss);
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? NAM_OK : cuda_fail((int)e, "log_l1: launch");
}
