// Encoder of the first training phase (Sec. 5.1): an MLP from the material
// parameters k(x) to the 8-channel latent, K -> 32 -> 32 -> 8 with ReLU
// hidden layers and a linear output.  It runs only in training: per query in
// the first phase (its output replaces the latent texture fetch) and once
// per texel to initialise the texture.
//
// Forward (encode_kernel): one thread per row, weights in shared memory.
// Backward (encoder_backward_kernel): a warp takes 32 rows; with a lane per row
// it recomputes the forward and back-propagates dL/dz, and between the layers,
// with a lane per block of a weight matrix, it sums that layer's outer products
// over the rows in registers.  Warps wait for none but themselves; their sums
// meet in shared memory, one atomic per parameter and CTA at the end.
// Both are bound by the latency of a row's chain of packed FMAs and shared
// loads at eight warps per SM, which the registers of fully unrolled layers
// leave (more warps with spilled registers were slower).  131,072 rows, four
// inputs: forward 19 us (a dot product per unit, 16 padded inputs: 32),
// backward 40 us (with tiles of 128 rows per CTA and barriers between a row
// phase and a block phase: 71).
#include <cuda_runtime.h>

#include <type_traits>

#include "nam_internal.h"
#include "tc_ptx.cuh"

namespace nam {
namespace {

constexpr int kE = 32;        // hidden width
constexpr int kKMax = 16;     // inputs, padded
constexpr int kBwdThreads = 128;
constexpr int kBwdCtas = 2;   // per SM

// Weights in shared memory, an input's weights side by side, so that one
// broadcast load feeds two packed FMAs on neighbouring units and the unit sums
// stay in registers (a dot product per unit took a load for every four FMAs).
// KP: inputs, padded to a multiple of four.
template <int KP>
struct EncW {
  float W1T[KP][kE];  // zero beyond K
  float b1[kE];
  float W2T[kE][kE];
  float b2[kE];
  float b3[8];
};

template <int KP>
__device__ void load_encoder(EncW<KP>& S, const float* __restrict__ p, int K, int t, int nt) {
  for (int i = t; i < kE * KP; i += nt) {
    const int j = i % kE, c = i / kE;
    S.W1T[c][j] = c < K ? p[j * K + c] : 0.0f;
  }
  p += kE * K;
  for (int i = t; i < kE; i += nt) S.b1[i] = p[i];
  p += kE;
  for (int i = t; i < kE * kE; i += nt) S.W2T[i % kE][i / kE] = p[i];
  p += kE * kE;
  for (int i = t; i < kE; i += nt) S.b2[i] = p[i];
  p += kE + 8 * kE;
  for (int i = t; i < 8; i += nt) S.b3[i] = p[i];
}

template <int KP>
__device__ __forceinline__ void load_row(const float* __restrict__ attrs, int K, int64_t i, float k[KP]) {
#pragma unroll
  for (int c = 0; c < KP; ++c) k[c] = c < K ? attrs[i * K + c] : 0.0f;
}

// acc[0..U) += w[0..U) x, w in shared memory
template <int U>
__device__ __forceinline__ void axpy(float2 (&acc)[U / 2], const float* w, float x) {
  const float2 xx = make_float2(x, x);
#pragma unroll
  for (int u = 0; u < U; u += 4) {
    const float4 v = *reinterpret_cast<const float4*>(w + u);
    acc[u / 2] = ptx::fma2(make_float2(v.x, v.y), xx, acc[u / 2]);
    acc[u / 2 + 1] = ptx::fma2(make_float2(v.z, v.w), xx, acc[u / 2 + 1]);
  }
}
template <int U>
__device__ __forceinline__ void start(float2 (&acc)[U / 2], const float* b) {
#pragma unroll
  for (int u = 0; u < U; u += 2) acc[u / 2] = *reinterpret_cast<const float2*>(b + u);
}
__device__ __forceinline__ uint32_t relu(float2 (&a)[kE / 2]) {
  uint32_t m = 0;
#pragma unroll
  for (int u = 0; u < kE / 2; ++u) {
    if (a[u].x > 0.0f) m |= 1u << (2 * u);
    if (a[u].y > 0.0f) m |= 2u << (2 * u);
    a[u] = make_float2(fmaxf(a[u].x, 0.0f), fmaxf(a[u].y, 0.0f));
  }
  return m;
}
__device__ __forceinline__ float unit(const float2 (&a)[kE / 2], int j) { return j & 1 ? a[j / 2].y : a[j / 2].x; }

// h1 = ReLU(W1 k + b1), h2 = ReLU(W2 h1 + b2); pre-activation signs in masks
template <int KP>
__device__ __forceinline__ void hidden(const EncW<KP>& S, const float k[KP], float2 (&h1)[kE / 2],
                                       float2 (&h2)[kE / 2], uint32_t& m1, uint32_t& m2) {
  start<kE>(h1, S.b1);
#pragma unroll
  for (int c = 0; c < KP; ++c) axpy<kE>(h1, S.W1T[c], k[c]);
  m1 = relu(h1);
  start<kE>(h2, S.b2);
#pragma unroll
  for (int c = 0; c < kE; ++c) axpy<kE>(h2, S.W2T[c], unit(h1, c));
  m2 = relu(h2);
}

constexpr int kFwdThreads = 128;
constexpr int kFwdCtas = 2;  // per SM

template <int KP>
__global__ void __launch_bounds__(kFwdThreads, kFwdCtas) encode_kernel(const float* __restrict__ W, int K,
                                                             const float* __restrict__ attrs, int64_t n,
                                                             float* __restrict__ z_out) {
  __shared__ __align__(16) EncW<KP> S;
  __shared__ __align__(16) float W3T[kE][8];
  load_encoder(S, W, K, threadIdx.x, blockDim.x);
  const float* W3 = W + kE * (K + 1) + kE * (kE + 1);
  for (int i = threadIdx.x; i < 8 * kE; i += blockDim.x) W3T[i % kE][i / kE] = W3[i];
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float k[KP];
    float2 h1[kE / 2], h2[kE / 2], z[4];
    uint32_t m1, m2;
    load_row<KP>(attrs, K, i, k);
    hidden(S, k, h1, h2, m1, m2);
    start<8>(z, S.b3);
#pragma unroll
    for (int j = 0; j < kE; ++j) axpy<8>(z, W3T[j], unit(h2, j));
    float4* o = reinterpret_cast<float4*>(z_out + i * 8);
    o[0] = make_float4(z[0].x, z[0].y, z[1].x, z[1].y);
    o[1] = make_float4(z[2].x, z[2].y, z[3].x, z[3].y);
  }
}

template <int KP>
struct EncBwdSmem {
  EncW<KP> w;
  float W2[kE][kE], W3[8][kE];
  // per warp, of its 32 rows (odd multiples of 16 bytes apart: no bank
  // conflicts): a layer's deltas, its inputs, dL/dz
  struct Warp {
    float D[32][kE + 4], X[32][kE + 4], DZ[32][8];
  } r[kBwdThreads / 32];
};

template <int KP>
__global__ void __launch_bounds__(kBwdThreads, kBwdCtas) encoder_backward_kernel(const float* __restrict__ W, int K,
                                                                 const float* __restrict__ attrs,
                                                                 const float* __restrict__ dz, int64_t n,
                                                                 float* __restrict__ grad,
                                                                 const int* __restrict__ failed) {
  if (failed && *failed) return;  // dz is not this batch's
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using Sm = EncBwdSmem<KP>;
  Sm& S = *reinterpret_cast<Sm*>(smem_raw);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  load_encoder(S.w, W, K, t, kBwdThreads);
  {
    const float* W2 = W + kE * (K + 1);
    for (int i = t; i < kE * kE; i += kBwdThreads) S.W2[i / kE][i % kE] = W2[i];
    for (int i = t; i < 8 * kE; i += kBwdThreads) S.W3[i / kE][i % kE] = W2[kE * (kE + 1) + i];
  }
  __syncthreads();
  typename Sm::Warp& R = S.r[warp];
  // this lane's gradients: dW3 rows 2r.., columns 4c..; dW2 rows 8r..,
  // columns 4c..; dW1 row `lane`; biases of unit `lane` (b3: lane % 8)
  const int r = lane >> 3, c = lane & 7;
  float2 acc3[4], acc2[16], acc1[KP / 2];
  float ab1 = 0.0f, ab2 = 0.0f, ab3 = 0.0f;
#pragma unroll
  for (int e = 0; e < 4; ++e) acc3[e] = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int e = 0; e < 16; ++e) acc2[e] = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int e = 0; e < KP / 2; ++e) acc1[e] = make_float2(0.0f, 0.0f);
  auto store = [&](float* row, const float2 (&v)[kE / 2]) {
#pragma unroll
    for (int j = 0; j < kE / 2; j += 2)
      reinterpret_cast<float4*>(row)[j / 2] = make_float4(v[j].x, v[j].y, v[j + 1].x, v[j + 1].y);
  };
  auto keep = [&](float2 (&v)[kE / 2], uint32_t m) {
#pragma unroll
    for (int u = 0; u < kE / 2; ++u)
      v[u] = make_float2((m >> (2 * u)) & 1u ? v[u].x : 0.0f, (m >> (2 * u + 1)) & 1u ? v[u].y : 0.0f);
  };
  // acc[2 rr .. 2 rr + 1] += d a
  auto outer = [&](float2* acc, int rr, float d, const float4& a) {
    const float2 dd = make_float2(d, d);
    acc[2 * rr] = ptx::fma2(dd, make_float2(a.x, a.y), acc[2 * rr]);
    acc[2 * rr + 1] = ptx::fma2(dd, make_float2(a.z, a.w), acc[2 * rr + 1]);
  };
  const int64_t ntiles = (n + 31) / 32;
  for (int64_t tile = blockIdx.x + (int64_t)warp * gridDim.x; tile < ntiles;
       tile += (int64_t)gridDim.x * (kBwdThreads / 32)) {
    const int64_t start_row = tile * 32;
    const int count = (int)((n - start_row) < 32 ? (n - start_row) : 32);
    const int64_t i = start_row + (lane < count ? lane : 0);
    // ---- lane = row: forward -------------------------------------------------
    float k[KP];
    float2 h1[kE / 2], h2[kE / 2];
    uint32_t m1, m2;
    load_row<KP>(attrs, K, i, k);
    const float4 ga = reinterpret_cast<const float4*>(dz + i * 8)[0];
    const float4 gb = reinterpret_cast<const float4*>(dz + i * 8)[1];
    hidden(S.w, k, h1, h2, m1, m2);
    store(R.X[lane], h2);
    reinterpret_cast<float4*>(R.DZ[lane])[0] = ga;
    reinterpret_cast<float4*>(R.DZ[lane])[1] = gb;
    __syncwarp();
    // ---- lane = block of dW3 -------------------------------------------------
#pragma unroll 4
    for (int q = 0; q < count; ++q) {
      const float2 d = *reinterpret_cast<const float2*>(&R.DZ[q][2 * r]);
      const float4 a = *reinterpret_cast<const float4*>(&R.X[q][4 * c]);
      outer(acc3, 0, d.x, a);
      outer(acc3, 1, d.y, a);
      ab3 += R.DZ[q][c];
    }
    // ---- lane = row: d2 = (W3^T dz) where layer 2 is active -------------------
    {
      const float g[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
#pragma unroll
      for (int u = 0; u < kE / 2; ++u) h2[u] = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int e = 0; e < 8; ++e) axpy<kE>(h2, S.W3[e], g[e]);
      keep(h2, m2);
    }
    __syncwarp();
    store(R.D[lane], h2);
    store(R.X[lane], h1);
    __syncwarp();
    // ---- lane = block of dW2 -------------------------------------------------
#pragma unroll 2
    for (int q = 0; q < count; ++q) {
      const float4 d0 = *reinterpret_cast<const float4*>(&R.D[q][8 * r]);
      const float4 d1 = *reinterpret_cast<const float4*>(&R.D[q][8 * r + 4]);
      const float4 a = *reinterpret_cast<const float4*>(&R.X[q][4 * c]);
      outer(acc2, 0, d0.x, a); outer(acc2, 1, d0.y, a); outer(acc2, 2, d0.z, a); outer(acc2, 3, d0.w, a);
      outer(acc2, 4, d1.x, a); outer(acc2, 5, d1.y, a); outer(acc2, 6, d1.z, a); outer(acc2, 7, d1.w, a);
      ab2 += R.D[q][lane];
    }
    // ---- lane = row: d1 = (W2^T d2) where layer 1 is active -------------------
#pragma unroll
    for (int u = 0; u < kE / 2; ++u) h1[u] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int j = 0; j < kE; ++j) axpy<kE>(h1, S.W2[j], unit(h2, j));
    keep(h1, m1);
    __syncwarp();
    store(R.D[lane], h1);
#pragma unroll
    for (int e = 0; e < KP / 4; ++e)
      reinterpret_cast<float4*>(R.X[lane])[e] = make_float4(k[4 * e], k[4 * e + 1], k[4 * e + 2], k[4 * e + 3]);
    __syncwarp();
    // ---- lane = row of dW1 ---------------------------------------------------
#pragma unroll 4
    for (int q = 0; q < count; ++q) {
      const float d = R.D[q][lane];
#pragma unroll
      for (int e = 0; e < KP / 4; ++e) outer(acc1, e, d, *reinterpret_cast<const float4*>(&R.X[q][4 * e]));
      ab1 += d;
    }
    __syncwarp();
  }
  // ---- the warps' sums meet in shared memory: one atomic per parameter and CTA
  const int ob1 = kE * K, oW2 = ob1 + kE, ob2 = oW2 + kE * kE, oW3 = ob2 + kE, ob3 = oW3 + 8 * kE, np = ob3 + 8;
  static_assert((kE * (KP + 1) + kE * (kE + 1) + 8 * (kE + 1)) * 4 <= (int)sizeof(typename Sm::Warp), "");
  float* o = reinterpret_cast<float*>(&R);
#pragma unroll
  for (int e = 0; e < KP; ++e)
    if (e < K) o[lane * K + e] = e & 1 ? acc1[e / 2].y : acc1[e / 2].x;
  o[ob1 + lane] = ab1;
  o[ob2 + lane] = ab2;
  if (lane < 8) o[ob3 + lane] = ab3;
#pragma unroll
  for (int rr = 0; rr < 8; ++rr)
#pragma unroll
    for (int e = 0; e < 4; ++e)
      o[oW2 + (8 * r + rr) * kE + 4 * c + e] = e & 1 ? acc2[2 * rr + e / 2].y : acc2[2 * rr + e / 2].x;
#pragma unroll
  for (int rr = 0; rr < 2; ++rr)
#pragma unroll
    for (int e = 0; e < 4; ++e)
      o[oW3 + (2 * r + rr) * kE + 4 * c + e] = e & 1 ? acc3[2 * rr + e / 2].y : acc3[2 * rr + e / 2].x;
  __syncthreads();
  for (int i = t; i < np; i += kBwdThreads) {
    float v = 0.0f;
#pragma unroll
    for (int w = 0; w < kBwdThreads / 32; ++w) v += reinterpret_cast<const float*>(&S.r[w])[i];
    atomicAdd(&grad[i], v);
  }
}

// the kernels for K inputs padded to 4, 8, 12 or 16 (padding to 16 always
// would be three quarters of the first layer's work for four inputs)
template <class F>
void by_inputs(int K, F&& f) {
  if (K <= 4) f(std::integral_constant<int, 4>());
  else if (K <= 8) f(std::integral_constant<int, 8>());
  else if (K <= 12) f(std::integral_constant<int, 12>());
  else f(std::integral_constant<int, 16>());
}

}  // namespace

int launch_encode(const float* W, int K, const float* attrs, int64_t n, float* z_out, int num_sms, void* stream) {
  if (n == 0) return 0;
  if (K < 1 || K > kKMax) return (int)cudaErrorInvalidValue;
  int64_t blocks = (n + kFwdThreads - 1) / kFwdThreads;
  const int64_t cap = (int64_t)num_sms * kFwdCtas;
  if (blocks > cap) blocks = cap;
  by_inputs(K, [&](auto kp) {
    encode_kernel<kp><<<(int)blocks, kFwdThreads, 0, (cudaStream_t)stream>>>(W, K, attrs, n, z_out);
  });
  return (int)cudaGetLastError();
}

int launch_encoder_backward(const float* W, int K, const float* attrs, const float* dz, int64_t n, float* grad,
                            int num_sms, const int* failed, void* stream) {
  if (n == 0) return 0;
  if (K < 1 || K > kKMax) return (int)cudaErrorInvalidValue;
  const int64_t tiles = (n + 31) / 32;  // one per warp
  int64_t grid = (int64_t)num_sms * kBwdCtas;
  if (grid > tiles) grid = tiles;
  by_inputs(K, [&](auto kp) {
    auto k = encoder_backward_kernel<kp>;
    const int smem = (int)sizeof(EncBwdSmem<kp>);
    static std::atomic<uint64_t> attr_done{0};
    once_per_device(attr_done, [&] { cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); });
    k<<<(int)grid, kBwdThreads, smem, (cudaStream_t)stream>>>(W, K, attrs, dz, n, grad, failed);
  });
  return (int)cudaGetLastError();
}

}  // namespace nam
