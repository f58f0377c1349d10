// Importance sampling with the neural proxy density (Sec. 4.3, Appendix A).
//
// Per query: latent fetch as for the BRDF, the sampler MLP 11 -> 32 -> 32 ->
// 32 -> 9 (ReLU hidden layers), the output activations, then either the
// mixture density of the query's wo or one sample of wo with its density.
// Sampler weights (FP32 masters) are laid out per layer as W (out x in) then
// b (out).
//
// The MLP runs on the tensor cores at FP32 accuracy, tiles of 128 queries as
// in the evaluation kernel: fetch warpgroups filter the latents and write
// layer 1's operand, chain warpgroups (thread r = query r = TMEM lane r) take
// a tile through the four layers.  Each weight is split into two binary16
// values, W = W_hi + W_lo, and each layer input into x = x_hi + x_lo (hi: x
// with its 13 low mantissa bits cleared, exact in binary16); one MMA over
// [x_hi | x_lo | 1 1] x [W_hi | W_hi | b_hi b_lo] and one over x_hi x W_lo give
// W x + b up to the dropped W_lo x_lo term, a relative 2^-22.  The proxy's
// activations, density and sampling run per thread in FP32.
// What bounds it: instruction issue (75 % of the slots); 1920x1080, sample and
// density: 97 us, 146 with the fetch in the chains' own warps.
#include <cuda_runtime.h>

#include "eval_tc.cuh"

namespace nam {

namespace {

constexpr float kPi = 3.14159265358979323846f;
constexpr float kAlphaMin = 1e-3f;
constexpr float kRhoMax = 0.99f;

__device__ __forceinline__ float qtanh(float x) {
  const float a = fabsf(x);
  return a >= 2.0f ? copysignf(1.0f, x) : x * (1.0f - 0.25f * a);
}
__device__ __forceinline__ float qsinh(float x) { return x * (1.0f + 0.5f * fabsf(x)); }

struct Proxy {
  float wd, mdx, mdy, ws, ax, ay, rho, msx, msy;
};

__device__ __forceinline__ Proxy activate(const float o[9]) {
  Proxy p;
  const float mx = fmaxf(o[0], o[3]);
  const float ed = expf(o[0] - mx), es = expf(o[3] - mx);
  const float inv = 1.0f / (ed + es);
  p.wd = ed * inv;
  p.ws = es * inv;
  p.mdx = qsinh(o[1]);
  p.mdy = qsinh(o[2]);
  p.ax = kAlphaMin + (1.0f - kAlphaMin) * 0.5f * (qtanh(o[4]) + 1.0f);
  p.ay = kAlphaMin + (1.0f - kAlphaMin) * 0.5f * (qtanh(o[5]) + 1.0f);
  p.rho = kRhoMax * qtanh(o[6]);
  p.msx = qsinh(o[7]);
  p.msy = qsinh(o[8]);
  return p;
}

// Half-vector density of the specular lobe: D_std(v / |v|) det(M^-1) / |v|^3,
// v = M^-1 h, D_std(w) = max(0, w_z) / pi.
__device__ __forceinline__ float pdf_half(const Proxy& p, float hx, float hy, float hz) {
  const float s = sqrtf(1.0f - p.rho * p.rho);
  const float vx = (hx + p.msx * hz) / p.ax;
  const float vy = (hy + p.msy * hz - p.ay * p.rho * vx) / (p.ay * s);
  const float vz = hz;
  const float vl2 = vx * vx + vy * vy + vz * vz;
  if (!(vz > 0.0f)) return 0.0f;
  // D_std(v/|v|) / |v|^3 = (vz / |v|) / pi / |v|^3 = vz / (pi |v|^4)
  return vz / (kPi * vl2 * vl2 * p.ax * p.ay * s);
}

__device__ __forceinline__ float pdf_full(const Proxy& p, const float wi[3], const float wo[3]) {
  const float ndx = -p.mdx, ndy = -p.mdy;
  const float ndl = rsqrtf(ndx * ndx + ndy * ndy + 1.0f);
  const float c = (wo[0] * ndx + wo[1] * ndy + wo[2]) * ndl;
  const float pd = c > 0.0f ? c / kPi : 0.0f;
  float hx = wi[0] + wo[0], hy = wi[1] + wo[1], hz = wi[2] + wo[2];
  const float hl2 = hx * hx + hy * hy + hz * hz;
  float ps = 0.0f;
  if (hl2 > 0.0f) {
    const float ih = rsqrtf(hl2);
    hx *= ih; hy *= ih; hz *= ih;
    const float oh = fabsf(wo[0] * hx + wo[1] * hy + wo[2] * hz);
    if (oh > 0.0f) ps = pdf_half(p, hx, hy, hz) / (4.0f * oh);
  }
  return p.wd * pd + p.ws * ps;
}

__device__ __forceinline__ void sample_dir(const Proxy& p, const float wi[3], float u0, float u1, float u2,
                                           float wo[3]) {
  const float r = sqrtf(u0);
  float sn, cs;
  sincospif(2.0f * u1, &sn, &cs);
  const float lx = r * cs, ly = r * sn, lz = sqrtf(fmaxf(1.0f - u0, 0.0f));
  if (u2 < p.wd) {
    // cosine lobe around n_d, frame from n_d by Duff et al.'s basis
    float n0 = -p.mdx, n1 = -p.mdy, n2 = 1.0f;
    const float il = rsqrtf(n0 * n0 + n1 * n1 + 1.0f);
    n0 *= il; n1 *= il; n2 *= il;
    const float sg = copysignf(1.0f, n2);
    const float a = -1.0f / (sg + n2);
    const float b = n0 * n1 * a;
    const float t0 = 1.0f + sg * n0 * n0 * a, t1 = sg * b, t2 = -sg * n0;
    const float b0 = n1 * t2 - n2 * t1, b1 = n2 * t0 - n0 * t2, b2 = n0 * t1 - n1 * t0;
    wo[0] = t0 * lx + b0 * ly + n0 * lz;
    wo[1] = t1 * lx + b1 * ly + n1 * lz;
    wo[2] = t2 * lx + b2 * ly + n2 * lz;
  } else {
    const float s = sqrtf(1.0f - p.rho * p.rho);
    float hx = p.ax * lx - p.msx * lz;
    float hy = p.ay * p.rho * lx + p.ay * s * ly - p.msy * lz;
    float hz = lz;
    const float ih = rsqrtf(hx * hx + hy * hy + hz * hz);
    hx *= ih; hy *= ih; hz *= ih;
    const float d = wi[0] * hx + wi[1] * hy + wi[2] * hz;
    wo[0] = 2.0f * d * hx - wi[0];
    wo[1] = 2.0f * d * hy - wi[1];
    wo[2] = 2.0f * d * hz - wi[2];
  }
}


// ---------------------------------------------------------------------------
// weight blob: MMA B operands in the canonical no-swizzle K-major layout
// (element (row, k) at (k / 8) * R * 16 + row * 16 + (k % 8) * 2 for an R-row
// block), rows = outputs:
//   A1 32 x 32  [W1_hi (11) b1_hi 0 0 0 0 | W1_hi (11) b1_lo 0 0 0 0]
//   L1 32 x 16  [W1_lo (11) 0 ...]
//   A2, A3 32 x 80  [W_hi (32) | W_hi (32) | b_hi b_lo 0 ...]
//   L2, L3 32 x 32  W_lo
//   A4, L4 as A2, L2 with 16 rows (9 used)
// ---------------------------------------------------------------------------
constexpr int kSA1 = 0, kSL1 = 2048, kSA2 = 3072, kSL2 = 8192, kSA3 = 10240, kSL3 = 15360, kSA4 = 17408,
              kSL4 = 19968, kSamplerBlobBytes = 20992;

// TMEM columns of one chain: the accumulator [0, 32), the A operand of layers
// 2 to 4 [32, 72): (h_hi, h_lo, 1 1 0 ...), the constant pair (1, 1) at
// column 64 written once.  Layer 1's operand comes from shared memory.
constexpr int kSD = 0, kSA = 32, kSCols = 72;

template <int NCH, int NF>
struct SamplerSmem {
  static constexpr int ZB = 8192;  // layer 1's operand: (x_hi, x_lo), 16 wide each, of 128 rows
  static constexpr int NZ = NCH % NF ? NCH * NF : NCH;  // as F16Smem::NZ
  static constexpr int Z_OFF = kSamplerBlobBytes;
  static constexpr int BAR_OFF = Z_OFF + NZ * ZB;
  static constexpr int BYTES = BAR_OFF + (NCH + 2 * NZ + 1) * 8 + 16;
};

template <bool F16P, int NCH, int NF>
__global__ void __launch_bounds__((NCH + NF) * 128, 1)
    sampler_tc_kernel(const __grid_constant__ LaunchCommon L, const uint8_t* __restrict__ blob, int mode,
                      const float* __restrict__ u, float* __restrict__ wo_out, float* __restrict__ pdf_out) {
  using S = SamplerSmem<NCH, NF>;
  constexpr int NZ = S::NZ;
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, r = tid & 127;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), wg = warp >> 2;
  const uint32_t aW = ptx::smem_u32(smem);
  const uint32_t bar0 = ptx::smem_u32(smem + S::BAR_OFF);
  const uint32_t bar_f = bar0 + 8 * NCH, bar_e = bar0 + 8 * (NCH + NZ), bar_w = bar0 + 8 * (NCH + 2 * NZ);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + S::BAR_OFF + (NCH + 2 * NZ + 1) * 8);

  if (tid == 0) {
    for (int k = 0; k < NCH; ++k) ptx::mbar_init(bar0 + 8 * k, 1);
    for (int k = 0; k < NZ; ++k) {
      ptx::mbar_init(bar_f + 8 * k, 4);  // the four warps of a fetch warpgroup
      ptx::mbar_init(bar_e + 8 * k, 1);
    }
    ptx::mbar_init(bar_w, 1);
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_u32(tslot), 512);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  constexpr uint32_t tmem = 0;  // all 512 columns are allocated

  const int64_t ntiles = (L.n + 127) / 128;
  const int64_t per = (ntiles + gridDim.x - 1) / gridDim.x;
  const int64_t c_begin = (int64_t)blockIdx.x * per;
  const int64_t c_end = c_begin + per < ntiles ? c_begin + per : ntiles;
  bool bad = *tslot != tmem, mma_pending = false, w_pending = false;
  uint32_t ph_m = 0;
  auto row_of = [&](const TileRef& t) -> int64_t { return t.start + (r < t.count ? r : 0); };

  if (wg >= NCH) {
    // ---- fetch: layer 1's input (z, wi, 1) as (hi, lo) -----------------------
    float wx, wy, wz;
    bad = !fetch_loop<F16P, false, !F16P, NF, NZ>(
        L, c_begin, c_end, wg - NCH, bar_f, bar_e, bad,
        [&](const TileRef&) { return reinterpret_cast<const uint8_t*>(L.pyr0); }, row_of,
        [&](const TileRef& t) {
          const int64_t i = row_of(t);
          wx = ptx::ld_nc_pinned(L.q.wix + i);
          wy = ptx::ld_nc_pinned(L.q.wiy + i);
          wz = ptx::ld_nc_pinned(L.q.wiz + i);
        },
        [&](int slot, const float z[8]) {
          uint32_t v[16];
#pragma unroll
          for (int j = 0; j < 4; ++j) split_pair<false>(z[2 * j], z[2 * j + 1], v[j], v[8 + j]);
          split_pair<false>(wx, wy, v[4], v[12]);
          split_pair<false>(wz, 1.0f, v[5], v[13]);
          v[13] = (v[13] & 0x0000FFFFu) | 0x3C000000u;  // lo block: the 1 meets b1_lo
          v[6] = v[7] = v[14] = v[15] = 0u;
          const uint32_t zs = aW + S::Z_OFF + slot * S::ZB + r * 16;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            ptx::st_shared_v4(zs + j * 2048, v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
          ptx::fence_proxy_async();
        });
  } else {
    // ---- chains ---------------------------------------------------------------
    const uint32_t bar_m = bar0 + 8 * wg, bar_id = 1 + wg;
    const uint32_t tB = tmem + wg * kSCols;
    const uint32_t tBl = tB + ((uint32_t)((warp & 3) * 32) << 16);
    if (tid == 0 && c_begin < c_end) {
      ptx::fence_proxy_async();
      ptx::mbar_arrive_expect_tx(bar_w, kSamplerBlobBytes);
      ptx::bulk_g2s(aW, blob, kSamplerBlobBytes, bar_w);
      w_pending = true;
    }
    {
      // the constant pair (1, 1) that meets the bias columns (b_hi, b_lo)
      uint32_t one[8] = {0x3C003C00u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
      ptx::tmem_st8(tBl + kSA + 32, one);
    }
    constexpr uint32_t ID32 = ptx::idesc_f16(128, 32);
    constexpr uint32_t ID16 = ptx::idesc_f16(128, 16);
    auto leader = [&]() -> bool { return ((warp ^ wg) & 3) == 0 && ptx::elect(); };

    auto stage_issue = [&](auto issue) -> bool {
      ptx::tmem_st_wait();
      ptx::tc_fence_before();
      if (ptx::bar_red_or(bar_id, 128, bad)) {
        bad = true;
        return false;
      }
      if (leader()) {
        ptx::tc_fence_after();
        issue();
        ptx::mma_commit(bar_m);
      }
      mma_pending = true;
      return true;
    };
    auto stage_wait = [&]() {
      bad |= !ptx::mbar_wait(bar_m, ph_m, L.timeout_ns);
      ph_m ^= 1;
      if (!bad) mma_pending = false;
      ptx::tc_fence_after();
    };
    // ReLU of the 32 accumulator columns, split into (h_hi, h_lo), 16 at a time
    auto hidden_operand = [&]() {
#pragma unroll
      for (int c0 = 0; c0 < 32; c0 += 16) {
        uint32_t acc[16];
        ptx::tmem_ld16(tBl + kSD + c0, acc);
        ptx::tmem_ld_wait();
        uint32_t hi[8], lo[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) split_pair<true>(f32_of(acc[2 * j]), f32_of(acc[2 * j + 1]), hi[j], lo[j]);
        ptx::tmem_st8(tBl + kSA + c0 / 2, hi);
        ptx::tmem_st8(tBl + kSA + 16 + c0 / 2, lo);
      }
    };
    // one hidden or output layer: [h_hi | h_lo | 1 1] x [W_hi | W_hi | b], then h_hi x W_lo
    auto layer_mmas = [&](int a_off, int l_off, int rows, uint32_t id) {
      const uint32_t lbo = (uint32_t)rows * 16, step = (uint32_t)rows * 32;
#pragma unroll
      for (int s = 0; s < 5; ++s)
        ptx::mma_f16_ts(tB + kSD, tB + kSA + 8 * s, ptx::sdesc(aW + a_off + s * step, lbo, 128), id, s > 0 ? 1u : 0u);
#pragma unroll
      for (int s = 0; s < 2; ++s)
        ptx::mma_f16_ts(tB + kSD, tB + kSA + 8 * s, ptx::sdesc(aW + l_off + s * step, lbo, 128), id, 1u);
    };

    int slot = wg;
    uint32_t ph_f = 0;
    bool w_ready = false;
    for (int64_t c = c_begin + wg; c < c_end; c += NCH) {
      const int64_t i_raw = c * 128 + r;
      const bool valid = i_raw < L.n;
      const int64_t i = valid ? i_raw : L.n - 1;
      if (!w_ready) {
        bad |= !ptx::mbar_wait(bar_w, 0, L.timeout_ns);
        if (!bad && tid == 0) w_pending = false;
        w_ready = true;
      }
      const uint32_t aZ = aW + S::Z_OFF + slot * S::ZB, be = bar_e + 8 * slot;
      bad |= !ptx::mbar_wait(bar_f + 8 * slot, ph_f, L.timeout_ns);
      slot += NCH;
      if (slot >= NZ) {
        slot -= NZ;
        ph_f ^= 1u;
      }
      if (!stage_issue([&] {
#pragma unroll
            for (int s = 0; s < 2; ++s)
              ptx::mma_f16(tB + kSD, ptx::sdesc(aZ + s * 4096, 2048, 128), ptx::sdesc(aW + kSA1 + s * 1024, 512, 128),
                           ID32, s > 0 ? 1u : 0u);
            ptx::mma_f16(tB + kSD, ptx::sdesc(aZ, 2048, 128), ptx::sdesc(aW + kSL1, 512, 128), ID32, 1u);
            ptx::mma_commit(be);
          }))
        break;
      const float wi[3] = {ptx::ld_nc_pinned(L.q.wix + i), ptx::ld_nc_pinned(L.q.wiy + i),
                           ptx::ld_nc_pinned(L.q.wiz + i)};
      stage_wait();
      // ---- layers 2, 3 (32 -> 32) and 4 (32 -> 9) -----------------------------
      hidden_operand();
      if (!stage_issue([&] { layer_mmas(kSA2, kSL2, 32, ID32); })) break;
      stage_wait();
      hidden_operand();
      if (!stage_issue([&] { layer_mmas(kSA3, kSL3, 32, ID32); })) break;
      stage_wait();
      hidden_operand();
      if (!stage_issue([&] { layer_mmas(kSA4, kSL4, 16, ID16); })) break;
      stage_wait();
      // ---- proxy parameters, density or sample --------------------------------
      float o[9];
      {
        uint32_t acc[16];
        ptx::tmem_ld16(tBl + kSD, acc);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 9; ++j) o[j] = f32_of(acc[j]);
      }
      ptx::tc_fence_before();
      if (valid) {
        const Proxy p = activate(o);
        if (mode == 0) {
          const float wo[3] = {L.q.wox[i], L.q.woy[i], L.q.woz[i]};
          pdf_out[i] = pdf_full(p, wi, wo);
        } else {
          float wo[3];
          sample_dir(p, wi, u[3 * i], u[3 * i + 1], u[3 * i + 2], wo);
          wo_out[3 * i] = wo[0];
          wo_out[3 * i + 1] = wo[1];
          wo_out[3 * i + 2] = wo[2];
          if (pdf_out) pdf_out[i] = pdf_full(p, wi, wo);
        }
      }
    }
  }

  // ---- teardown (as in the evaluation kernel) --------------------------------
  bool drained = true;
  if (r == 0 && mma_pending) drained &= ptx::mbar_wait(bar0 + 8 * wg, ph_m ^ 1, ptx::kDrainTimeoutNs);
  if (tid == 0 && w_pending) drained &= ptx::mbar_wait(bar_w, 0, ptx::kDrainTimeoutNs);
  if (bad) record_error(L.err, DEVERR_WAIT_TIMEOUT);
  if (!drained) record_error(L.err, DEVERR_DRAIN_TIMEOUT);
  ptx::tc_fence_before();
  const bool all_drained = __syncthreads_and(drained ? 1 : 0) != 0;
  if (warp == 0 && all_drained) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(*tslot, 512);
  }
}

}  // namespace

size_t sampler_blob_bytes() { return (size_t)kSamplerBlobBytes; }

// x = hi + lo in binary16: hi = x with its 13 low mantissa bits cleared
// (rounded to binary16, exact over its normal range), lo = the rest rounded
// to binary16.
static void split_f16(float x, __half& hi, __half& lo) {
  uint32_t b;
  std::memcpy(&b, &x, 4);
  b &= 0xFFFFE000u;
  float t;
  std::memcpy(&t, &b, 4);
  hi = __float2half_rn(t);
  lo = __float2half_rn(x - __half2float(hi));
}

static void put_half(uint8_t* base, int R, int row, int k, __half h) {
  std::memcpy(base + (k / 8) * (R * 16) + row * 16 + (k % 8) * 2, &h, 2);
}

int pack_sampler_blob(const float* w, uint8_t* out) {
  for (int i = 0; i < kSamplerFloats; ++i)
    if (!(std::fabs(w[i]) < 32768.0f)) return -1;  // beyond the binary16 split
  std::memset(out, 0, kSamplerBlobBytes);
  const float* W1 = w;
  const float* b1 = W1 + 11 * 32;
  __half hi, lo;
  for (int j = 0; j < 32; ++j) {
    for (int k = 0; k < 11; ++k) {
      split_f16(W1[j * 11 + k], hi, lo);
      put_half(out + kSA1, 32, j, k, hi);
      put_half(out + kSA1, 32, j, 16 + k, hi);
      put_half(out + kSL1, 32, j, k, lo);
    }
    split_f16(b1[j], hi, lo);
    put_half(out + kSA1, 32, j, 11, hi);
    put_half(out + kSA1, 32, j, 27, lo);
  }
  // layers 2..4: W (rows x 32) then b
  const float* p = b1 + 32;
  const int a_off[3] = {kSA2, kSA3, kSA4}, l_off[3] = {kSL2, kSL3, kSL4}, rows[3] = {32, 32, 9};
  for (int l = 0; l < 3; ++l) {
    const int R = l < 2 ? 32 : 16;
    const float* W = p;
    const float* b = W + rows[l] * 32;
    for (int j = 0; j < rows[l]; ++j) {
      for (int k = 0; k < 32; ++k) {
        split_f16(W[j * 32 + k], hi, lo);
        put_half(out + a_off[l], R, j, k, hi);
        put_half(out + a_off[l], R, j, 32 + k, hi);
        put_half(out + l_off[l], R, j, k, lo);
      }
      split_f16(b[j], hi, lo);
      put_half(out + a_off[l], R, j, 64, hi);
      put_half(out + a_off[l], R, j, 65, lo);
    }
    p = b + rows[l];
  }
  return 0;
}

template <bool F16P>
static int launch_sampler_tc(const LaunchCommon& L, const void* blob, int mode, const float* u, float* wo_out,
                             float* pdf_out, cudaStream_t s) {
  // six chains (TMEM 6 x 72 columns) and two fetch warpgroups, 1024 threads at
  // <= 64 registers (1920x1080, sample and density: 97 us; 5 + 2 99, 4 + 2 109)
  constexpr int NCH = 6, NF = 2;
  using S = SamplerSmem<NCH, NF>;
  static_assert(S::BYTES <= 227 * 1024, "shared memory");
  static_assert(NCH * kSCols <= 512, "TMEM columns");
  auto k = sampler_tc_kernel<F16P, NCH, NF>;
  static std::atomic<uint64_t> configured{0};
  once_per_device(configured, [&] {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, S::BYTES);
    const int pct = (S::BYTES + 1024) * 100 / (228 * 1024) + 1;
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
  });
  const int64_t ntiles = (L.n + 127) / 128;
  const int grid = (int)(ntiles < L.num_sms ? ntiles : L.num_sms);
  k<<<grid, (NCH + NF) * 128, S::BYTES, s>>>(L, reinterpret_cast<const uint8_t*>(blob), mode, u, wo_out, pdf_out);
  return (int)cudaGetLastError();
}

int launch_sampler(const LaunchCommon& L, const void* blob, int mode, const float* u, float* wo_out,
                   float* pdf_out, void* stream) {
  if (L.n == 0) return 0;
  cudaStream_t s = (cudaStream_t)stream;
  return L.pyr.f16 ? launch_sampler_tc<true>(L, blob, mode, u, wo_out, pdf_out, s)
                   : launch_sampler_tc<false>(L, blob, mode, u, wo_out, pdf_out, s);
}

}  // namespace nam
