// FP16 tensor-core evaluation of the neural BRDF on sm_103a (tcgen05 + TMEM),
// pipelined over 128-query tiles.
//
// One CTA per SM.  "Fetch" warpgroups gather and filter the latents of the
// CTA's tiles (128 queries each); a "chain" warpgroup owns a tile at a time
// (thread r = query r = TMEM lane r) and takes it through the MMA stages on
// its own TMEM columns:
//   1. latent z (Sec. 4.1, trilinear or stochastic filtering of the pyramid,
//      FP32 filter), left in shared memory by a fetch warpgroup -> MMA 1: the
//      frame layer (Sec. 4.2) and the z part of decoder layer 1 share their
//      input, so one MMA of N = 16 + H computes both;
//   2. the frame MLP's second layer (8 -> 16 -> 6 form);
//   3. frame build (Gram-Schmidt, b = n x t) and the direction transform
//      (Eq. 4) in FP32 registers -> MMA 3 adds the direction part of decoder
//      layer 1 and its bias onto MMA 1's accumulator;
//   4. hidden layers (ReLU, FP16 operands);
//   5. output layer in FP32 on the FMA pipes, RGB store (x max(0, wi.z) if
//      asked, Eq. 1).
// Precision: FP16 weights (post-training quantised, Sec. 5.2), FP32
// accumulation.  z, the transformed directions and the frame MLP's hidden
// layer (every hidden layer for H < 64) enter the MMA as two FP16 halves (x =
// hi + lo, hi = x with its 13 low mantissa bits cleared, exact in FP16; lo =
// x - hi, rounded), i.e. at ~22-bit accuracy; the other hidden layers are
// rounded to FP16 once; the output layer reads the last one in FP32.
// What bounds it (1920x1080, H = 64): instruction issue (1,028 thread
// instructions per query, 70 % of the issue slots) and the chain of MMA round
// trips.  Measured on the way, 1920x1080: 117 us with the fetch in the
// chains' own warps through cp.async, 112 with fetch warps staging through
// cp.async, 111 with the texels in their registers, 98 with the output layer
// on the FMA pipes (its operand split and MMA round trip cost more than its
// 96 packed FMAs with weights from constant memory; from shared memory they
// make the frame 117 us, since the gathers keep the load/store pipe busy), 89
// with MMA issue spread over the schedulers and a constant TMEM base.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace nam {

// ---------------------------------------------------------------------------
// weight blob: MMA B operands (rows = N = outputs, K = inputs), canonical
// no-swizzle K-major layout (8-row x 16-byte core matrices: element (row, k)
// at (k / 8) * (R * 16) + row * 16 + (k % 8) * 2 for an R-row block)
// ---------------------------------------------------------------------------
struct F16Lay {
  int NF;     // frame rows in the first MMA: 16 (frame forms 1, 2) or 0
  int N1;     // first MMA's N: H rows of decoder layer 1 (z inputs), then NF
  int ND;     // direction inputs of decoder layer 1: 6, or 12 (paper form)
  int KD;     // K of the direction block: (dir hi, dir lo, 1, 0 ...)
  int B1;     // N1 x 16: [W(z) | W(z)] for the operand (z hi, z lo)
  int B1B;    // 16 x 16: frame-layer bias in column 0 (A = constant block)
  int BF2;    // form 1: 16 x 32: [Wf2 | Wf2] (6 rows used)
  int BD;     // H x KD: [W(dirs) | W(dirs) | b1 | 0 ..]
  int BH;     // NH - 1 blocks of H x (H + 16): [W | b 0 ..]
  // FP32 (binary16-rounded values):
  int SB;     // [0, 8): FP8 scales; [8, 14): frame MLP layer 2's bias; [16, 22): output bias
  int WO;     // output layer, [6 outputs][H], halved (NarrowW)
  int BYTES;
};

__host__ __device__ constexpr F16Lay f16_lay(int H, int FK, int NH) {
  F16Lay o{};
  o.NF = FK ? 16 : 0;
  o.N1 = H + o.NF;
  o.ND = FK == 2 ? 12 : 6;
  o.KD = FK == 2 ? 32 : 16;
  o.B1 = 0;
  o.B1B = o.B1 + o.N1 * 16 * 2;
  o.BF2 = o.B1B + (FK ? 16 * 16 * 2 : 0);
  o.BD = o.BF2 + (FK == 1 ? 16 * 32 * 2 : 0);
  o.BH = o.BD + H * o.KD * 2;
  o.SB = o.BH + (NH - 1) * H * (H + 16) * 2;
  o.WO = o.SB + 24 * 4;
  o.BYTES = o.WO + 6 * H * 4;
  return o;
}

static inline bool f16_supported(const Shape& s) {
  const bool hidden_ok = (s.NH == 2 && (s.H == 16 || s.H == 32 || s.H == 64)) || (s.NH == 3 && s.H == 64);
  return hidden_ok && s.frame >= 0 && s.frame <= 2 && (s.out == 3 || s.out == 6);
}

// ---------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ float f32_of(uint32_t x) { return __uint_as_float(x); }

// x = hi + lo with hi = x whose 13 low mantissa bits are cleared (at most 11
// significant bits: exact in binary16 over its normal range) and lo = x - hi
// (exact in FP32, then rounded to binary16: |error| <= 2^-21 |x|).  hi and lo
// carry the sign of x, so with RELU both halves of a negative x become +0.
template <bool RELU>
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& hi, uint32_t& lo) {
  const float ta = __uint_as_float(__float_as_uint(a) & 0xFFFFE000u);
  const float tb = __uint_as_float(__float_as_uint(b) & 0xFFFFE000u);
  const float2 d = ptx::sub2(make_float2(a, b), make_float2(ta, tb));
  if (RELU) {
    hi = ptx::pack_h2_relu(ta, tb);
    lo = ptx::pack_h2_relu(d.x, d.y);
  } else {
    hi = ptx::pack_h2(ta, tb);
    lo = ptx::pack_h2(d.x, d.y);
  }
}

// The fetch-side query fields, loaded two tiles ahead of their use.
struct QF {
  float u, v, lod, xi;
};
// A query field.  Queries read through a permutation (GATHER) share their
// sectors with queries of other tiles and stay in L1; others are read once.
template <bool GATHER>
__device__ __forceinline__ float ld_field(const float* p) {
  return GATHER ? ptx::ld_nc_pinned(p) : ptx::ld_nc_stream(p);
}
template <bool GATHER>
__device__ __forceinline__ QF load_qf(const QueryPtrs& q, int64_t i) {
  QF x;
  x.u = ld_field<GATHER>(q.u + i);
  x.v = ld_field<GATHER>(q.v + i);
  x.lod = ld_field<GATHER>(q.lod + i);
  x.xi = q.xi ? ld_field<GATHER>(q.xi + i) : 0.0f;
  return x;
}

// A tile: up to 128 consecutive queries of one material.
struct TileRef {
  int64_t start;
  int count, mat;
};
__device__ __forceinline__ TileRef tile_at(const LaunchCommon& L, int64_t c) {
  TileRef t;
  if (L.chunks) {
    const Chunk ch = L.chunks[c];
    t.start = ch.start;
    t.count = ch.count;
    t.mat = ch.material;
  } else {
    t.start = c * 128;
    t.count = (int)((L.n - t.start) < 128 ? (L.n - t.start) : 128);
    t.mat = 0;
  }
  return t;
}

// Latent fetch of warps that do nothing else: the texels go through registers
// (no staging, the other warps hide the latency).  Bilinear taps of level l
// (Sec. 4.1; texel centres at (i + 1/2) / W): texel indices and weights wl *
// (bilinear weight).
// Power-of-two wrap, every lane's |u W0|, |v H0| < 2^22 - 1 (warp-uniform
// `fast`): floor(x) comes from one round-down addition of 1.5 2^23, whose
// result holds the integer in its low mantissa bits (no conversion
// instructions, which run at a quarter of the rate), and W_l, H_l from the
// exponents of level 0's sizes.
// EXACT: fractions and weights as in tap_axis and bilinear_acc, bit for bit.
template <bool EXACT>
__device__ __forceinline__ void level_taps(const PyrDesc& P, int l, float u, float v, bool fast, int lw0, int lh0,
                                           float wl, uint32_t idx[4], float* w) {
  int x0, x1, y0, y1, W;
  float fx, fy;
  if (fast) {
    const int ew = max(lw0 - l, 0), eh = max(lh0 - l, 0);
    const float X = u * __int_as_float((127 + ew) << 23), Y = v * __int_as_float((127 + eh) << 23);
    int kx, ky;
    if (EXACT) {
      // the 1/2 comes off the fractional part (tap_axis)
      const float tx = __fadd_rd(X, 12582912.0f), ty = __fadd_rd(Y, 12582912.0f);
      const float rx = X - (tx - 12582912.0f), ry = Y - (ty - 12582912.0f);
      kx = __float_as_int(tx) - (rx >= 0.5f ? 0 : 1);
      ky = __float_as_int(ty) - (ry >= 0.5f ? 0 : 1);
      fx = rx >= 0.5f ? rx - 0.5f : rx + 0.5f;
      fy = ry >= 0.5f ? ry - 0.5f : ry + 0.5f;
    } else {
      const float xs = X - 0.5f, ys = Y - 0.5f;
      const float tx = __fadd_rd(xs, 12582912.0f), ty = __fadd_rd(ys, 12582912.0f);
      fx = xs - (tx - 12582912.0f);
      fy = ys - (ty - 12582912.0f);
      kx = __float_as_int(tx);
      ky = __float_as_int(ty);
    }
    W = 1 << ew;
    const int mx = W - 1, my = (1 << eh) - 1;
    x0 = kx & mx;
    x1 = (kx + 1) & mx;
    y0 = ky & my;
    y1 = (ky + 1) & my;
  } else {
    W = P.w[l];
    tap_axis(P, u, W, x0, x1, fx);
    tap_axis(P, v, P.h[l], y0, y1, fy);
  }
  const uint32_t base = (uint32_t)P.off[l];
  const uint32_t r0 = base + (uint32_t)y0 * (uint32_t)W, r1 = base + (uint32_t)y1 * (uint32_t)W;
  const float gx = 1.0f - fx, gy = 1.0f - fy;
  if (EXACT) {
    w[0] = gx * gy * wl;
    w[1] = fx * gy * wl;
    w[2] = gx * fy * wl;
    w[3] = fx * fy * wl;
  } else {
    const float a = gy * wl, b = fy * wl;
    w[0] = gx * a;
    w[1] = fx * a;
    w[2] = gx * b;
    w[3] = fx * b;
  }
  idx[0] = r0 + x0;
  idx[1] = r0 + x1;
  idx[2] = r1 + x0;
  idx[3] = r1 + x1;
}

// acc += sum_k w_k texel_k over one level's four taps, in FP32
template <bool F16P>
__device__ __forceinline__ void filter4(const uint4 (&t)[F16P ? 4 : 8], const float* w, float2 acc[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 wk = make_float2(w[k], w[k]);
    if constexpr (F16P) {
      const __half2* h = reinterpret_cast<const __half2*>(&t[k]);
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[c] = ptx::fma2(wk, __half22float2(h[c]), acc[c]);
    } else {
      const uint4 a = t[2 * k], b = t[2 * k + 1];
      acc[0] = ptx::fma2(wk, make_float2(f32_of(a.x), f32_of(a.y)), acc[0]);
      acc[1] = ptx::fma2(wk, make_float2(f32_of(a.z), f32_of(a.w)), acc[1]);
      acc[2] = ptx::fma2(wk, make_float2(f32_of(b.x), f32_of(b.y)), acc[2]);
      acc[3] = ptx::fma2(wk, make_float2(f32_of(b.z), f32_of(b.w)), acc[3]);
    }
  }
}

template <bool F16P>
__device__ __forceinline__ void load4(const uint8_t* pyr, const uint32_t idx[4], uint4 (&t)[F16P ? 4 : 8]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint4* p = reinterpret_cast<const uint4*>(pyr + (size_t)idx[k] * (F16P ? 16 : 32));
    if constexpr (F16P) {
      t[k] = __ldg(p);
    } else {
      t[2 * k] = __ldg(p);
      t[2 * k + 1] = __ldg(p + 1);
    }
  }
}

// z of one query (Sec. 4.1): levels l0 (weight 1 - t) and l1 (weight t; not
// read when t = 0), or the stochastic pick of one of them.
template <bool F16P, bool EXACT>
__device__ __forceinline__ void fetch_direct(const PyrDesc& P, const uint8_t* pyr, const QF& q, int lw0, int lh0,
                                             float z[8]) {
  const float l = fminf(fmaxf(q.lod, 0.0f), (float)(P.levels - 1));  // NaN -> 0
  const float fl = floorf(l);
  const int l0 = (int)fl;
  const int l1 = min(l0 + 1, P.levels - 1);
  const float t = l - fl;
  const bool stoch = P.filter == NAM_FILTER_STOCHASTIC;
  const int la = stoch && q.xi < t ? l1 : l0;
  const bool in_range = fabsf(q.u * (float)P.w[0]) < 4194303.0f && fabsf(q.v * (float)P.h[0]) < 4194303.0f;
  const bool fast = P.pow2 && P.address == NAM_ADDRESS_WRAP && __all_sync(0xffffffffu, in_range);
  float2 acc[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) acc[c] = make_float2(0.0f, 0.0f);
  uint32_t idx[4];
  float wa[4];
  uint4 ta[F16P ? 4 : 8];
  level_taps<EXACT>(P, la, q.u, q.v, fast, lw0, lh0, stoch ? 1.0f : 1.0f - t, idx, wa);
  load4<F16P>(pyr, idx, ta);
  if (!stoch) {
    float wb[4];
    uint4 tb[F16P ? 4 : 8];
    level_taps<EXACT>(P, l1, q.u, q.v, fast, lw0, lh0, t, idx, wb);
    if (t != 0.0f) {
      load4<F16P>(pyr, idx, tb);
    } else {
#pragma unroll
      for (int k = 0; k < (F16P ? 4 : 8); ++k) tb[k] = make_uint4(0u, 0u, 0u, 0u);
    }
    filter4<F16P>(ta, wa, acc);
    filter4<F16P>(tb, wb, acc);
  } else {
    filter4<F16P>(ta, wa, acc);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    z[2 * c] = acc[c].x;
    z[2 * c + 1] = acc[c].y;
  }
}

// The loop of one fetch warpgroup (fw of NF): it takes tiles fw, fw + NF, ...
// of the CTA's range [c_begin, c_end), each warp its own 32 rows, and hands
// tile t's filtered latents to the chains through ring entry t % NZ:
// begin(tile) may start loads of its own, emit(slot, z) writes this row's;
// bar_f[slot] counts the four warps that
// filled it, bar_e[slot] its reading.  The next tile's query fields are in
// flight while this tile's texels are.  False if a wait ran out.
template <bool F16P, bool MULTI, bool EXACT, int NF, int NZ, class PyrFor, class RowOf, class Begin, class Emit>
__device__ __forceinline__ bool fetch_loop(const LaunchCommon& L, int64_t c_begin, int64_t c_end, int fw, uint32_t bar_f,
                                           uint32_t bar_e, bool bad, PyrFor pyr_for, RowOf row_of, Begin begin,
                                           Emit emit) {
  const int lw0 = 31 - __clz(L.pyr.w[0]), lh0 = 31 - __clz(L.pyr.h[0]);
  int64_t c = c_begin + fw;
  int slot = fw, pass = 0;
  TileRef nxt{};
  QF qn{};
  if (c < c_end) {
    nxt = tile_at(L, c);
    if (nxt.count > 0) qn = load_qf<MULTI>(L.q, row_of(nxt));
  }
  for (; c < c_end; c += NF) {
    const TileRef cur = nxt;
    const QF q = qn;
    if (c + NF < c_end) {
      nxt = tile_at(L, c + NF);
      if (nxt.count > 0) qn = load_qf<MULTI>(L.q, row_of(nxt));
    }
    if (cur.count > 0) begin(cur);
    float z[8];
    if (cur.count > 0) fetch_direct<F16P, EXACT>(L.pyr, pyr_for(cur), q, lw0, lh0, z);
    // the entry's previous latents have been read
    if (pass > 0) bad |= !ptx::mbar_wait(bar_e + 8 * slot, (uint32_t)(pass - 1) & 1u, L.timeout_ns);
    if (__any_sync(0xffffffffu, bad)) return false;
    if (cur.count > 0) emit(slot, z);
    __syncwarp();
    if ((threadIdx.x & 31) == 0) ptx::mbar_arrive(bar_f + 8 * slot);
    slot += NF;
    if (slot >= NZ) {
      slot -= NZ;
      ++pass;
    }
  }
  return true;
}

// ---------------------------------------------------------------------------
// kernel
// ---------------------------------------------------------------------------
// A launch that mixes materials keeps this many weight slots per CTA, shared
// by its warpgroups: a warpgroup whose tile needs a material finds it in a
// slot, or loads it into a slot no warpgroup is using.
constexpr int kMultiSlots = 2;

// Warpgroups of a CTA (one CTA per SM): NCH "chain" warpgroups take one tile
// each through the MMA stages; NF "fetch" warpgroups gather and filter the
// latents and leave each tile's first operand in shared memory.  A tile's
// chain is a sequence of MMA round trips with idle issue slots between them;
// with the fetch (a third of a query's instructions and its longest memory
// wait) in warps of its own, seven warpgroups are in flight instead of five
// (TMEM holds at most five chains at H = 64) and the chain is shorter.

// Shared memory: constant block (1.0 in column 0 of every row) and zero block
// (the A operand of the bias steps), the weight slots (one, or kMultiSlots
// when a launch mixes materials), the latent operands (tile t's in buffer
// t % NZ), the mbarriers (per chain its MMAs, per operand full and read, per weight slot its loads), the TMEM
// address, then the slot table: per slot its material, users and load count,
// a lock, and one word per chain to broadcast the slot its leader acquired.
template <int H, int FK, int NH, bool F16P, bool MULTI, int NCH, int NF>
struct F16Smem {
  static constexpr F16Lay Y = f16_lay(H, FK, NH);
  static constexpr int SLOTS = MULTI ? kMultiSlots : 1;
  static constexpr int BLOB_AL = (Y.BYTES + 127) / 128 * 128;
  static constexpr int W_OFF = 4096;
  static constexpr int Z_OFF = W_OFF + SLOTS * BLOB_AL;
  static constexpr int ZB = 4096;  // (z hi, z lo): two 8-wide core columns of 128 rows
  // a multiple of both counts: a buffer is always filled by the same fetch
  // warpgroup and read by the same chain, so that each side has seen the
  // phase before the one it waits for (a wait by parity tells only
  // neighbouring phases apart)
  static constexpr int NZ = NCH % NF ? NCH * NF : NCH;
  static constexpr int BAR_OFF = Z_OFF + NZ * ZB;
  static constexpr int TSLOT_OFF = (BAR_OFF + 8 * (NCH + 2 * NZ + SLOTS) + 15) / 16 * 16;
  static constexpr int TAB_OFF = TSLOT_OFF + 16;
  static constexpr int BYTES = (TAB_OFF + 4 * (3 * SLOTS + 1 + NCH) + 15) / 16 * 16;
};

// A lock word in shared memory, taken with a time limit (false: not taken).
__device__ __forceinline__ bool smem_lock(int* l, uint64_t t0, uint64_t timeout_ns) {
  while (atomicCAS(l, 0, 1) != 0) {
    if (ptx::globaltimer() - t0 > timeout_ns) return false;
    __nanosleep(64);
  }
  __threadfence_block();
  return true;
}
__device__ __forceinline__ void smem_unlock(int* l) {
  __threadfence_block();
  atomicExch(l, 0);
}

// TMEM columns of one chain (H + 32):
//   [0, H)        decoder accumulator (layer 1, hidden layers)
//   [H, H + 16)   frame-layer accumulator; later the hidden-layer operand
//                 [H, H + H/2) (FP16 pairs)
//   [H+16, H+32)  operands of the frame MLP's second layer, directions
template <int H>
struct F16Cols {
  static constexpr int COLS = H + 32;
  static constexpr int D = 0, F = H, A = H + 16, HID = H;
};

// The output layer's weights as kernel parameters (NarrowW, rows of H); empty
// when the launch mixes materials.
template <int H, bool MULTI>
struct OutParams {
  float wo[6][H], bo[6];
};
template <int H>
struct OutParams<H, true> {};

template <int H, int FK, int NH, bool F16P, bool MULTI, int NCH, int NF, bool P8>
__global__ void __launch_bounds__((NCH + NF) * 128, 1) eval_f16_kernel(const __grid_constant__ LaunchCommon L,
                                                                      const __grid_constant__ OutParams<H, MULTI> O) {
  static_assert(NF == 2 || NF == 3, "F16Smem::NZ is the least common multiple for a prime count");
  using S = F16Smem<H, FK, NH, F16P, MULTI, NCH, NF>;
  using C = F16Cols<H>;
  constexpr F16Lay Y = S::Y;
  constexpr int ND = Y.ND;
  extern __shared__ __align__(1024) uint8_t smem[];

  const int tid = threadIdx.x, r = tid & 127;
  // warp-uniform to the compiler too (addresses and descriptors of the MMAs
  // are then computed once per warp)
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), wg = warp >> 2;
  const uint32_t aConst = ptx::smem_u32(smem);
  uint32_t aW = ptx::smem_u32(smem + S::W_OFF);  // the weight slot this warpgroup reads
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S::BAR_OFF);
  const uint32_t bar0 = ptx::smem_u32(bars);
  constexpr int NZ = S::NZ;
  const uint32_t bar_f = bar0 + 8 * NCH;                 // operand k full
  const uint32_t bar_e = bar0 + 8 * (NCH + NZ);          // operand k read
  const uint32_t bar_w = bar0 + 8 * (NCH + 2 * NZ);      // weight slot k loaded
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + S::TSLOT_OFF);
  // slot table (mixed-material launches)
  volatile int* slot_mat = reinterpret_cast<volatile int*>(smem + S::TAB_OFF);
  volatile int* slot_users = slot_mat + S::SLOTS;
  volatile int* slot_loads = slot_users + S::SLOTS;
  int* slot_lock = const_cast<int*>(slot_loads + S::SLOTS);
  volatile int* wg_word = slot_loads + S::SLOTS + 1;

  if (tid == 0) {
    for (int k = 0; k < NCH; ++k) ptx::mbar_init(bar0 + 8 * k, 1);
    for (int k = 0; k < NZ; ++k) {
      ptx::mbar_init(bar_f + 8 * k, 4);  // the four warps of a fetch warpgroup
      ptx::mbar_init(bar_e + 8 * k, 1);
    }
    for (int k = 0; k < S::SLOTS; ++k) {
      ptx::mbar_init(bar_w + 8 * k, 1);
      slot_mat[k] = -1;
      slot_users[k] = 0;
      slot_loads[k] = 0;
    }
    *slot_lock = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_u32(tslot), 512);
    ptx::tmem_relinquish();
  }
  if (tid < 128) {
    ptx::st_shared_v4(aConst + tid * 16, 0x3C00u, 0u, 0u, 0u);
    ptx::st_shared_v4(aConst + 2048 + tid * 16, 0u, 0u, 0u, 0u);
  }
  ptx::fence_proxy_async();
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  // all 512 columns are allocated, so they start at 0: a constant base
  constexpr uint32_t tmem = 0;

  int64_t ntiles = L.chunks ? (int64_t)L.n_chunks : (L.n + 127) / 128;
  if (L.n_chunks_dev) {
    const int64_t d = *L.n_chunks_dev;  // written by an earlier launch on this stream
    ntiles = d < 0 ? 0 : d < ntiles ? d : ntiles;
  }
  const int64_t per = (ntiles + gridDim.x - 1) / gridDim.x;
  const int64_t c_begin = (int64_t)blockIdx.x * per;
  const int64_t c_end = c_begin + per < ntiles ? c_begin + per : ntiles;

  bool bad = *tslot != tmem, mma_pending = false, w_pending = false;
  uint32_t ph_m = 0;
  int my_slot = -1;
  // the query behind row k of the chunk table (binned launches read the
  // caller's arrays through the binning permutation)
  auto src = [&](int64_t k) -> int64_t {
    if constexpr (MULTI) {
      if (L.gather) return (int64_t)__ldg(L.gather + k);
    }
    return k;
  };
  auto row_of = [&](const TileRef& t) -> int64_t { return src(t.start + (r < t.count ? r : 0)); };

  if (wg >= NCH) {
    auto pyr_for = [&](const TileRef& t) -> const uint8_t* {
      return reinterpret_cast<const uint8_t*>(MULTI ? L.mats.pyramid[t.mat] : L.pyr0);
    };
    // (FP32 texels: bilinear_acc's operation order)
    bad = !fetch_loop<F16P, MULTI, !F16P, NF, NZ>(
        L, c_begin, c_end, wg - NCH, bar_f, bar_e, bad, pyr_for, row_of, [](const TileRef&) {},
        [&](int slot, const float z[8]) {
          uint32_t v[8];
          split_pair<false>(z[0], z[1], v[0], v[4]);
          split_pair<false>(z[2], z[3], v[1], v[5]);
          split_pair<false>(z[4], z[5], v[2], v[6]);
          split_pair<false>(z[6], z[7], v[3], v[7]);
          const uint32_t zs = ptx::smem_u32(smem + S::Z_OFF) + slot * S::ZB + r * 16;
          ptx::st_shared_v4(zs, v[0], v[1], v[2], v[3]);         // z hi
          ptx::st_shared_v4(zs + 2048, v[4], v[5], v[6], v[7]);  // z lo
          ptx::fence_proxy_async();
        });
  } else {
  // ========================= chain warpgroups ==============================
  const uint32_t bar_m = bar0 + 8 * wg;
  const uint32_t bar_id = 1 + wg;  // named barrier of this warpgroup
  const uint32_t tB = tmem + wg * C::COLS;                        // MMA addresses (lane 0)
  const uint32_t tBl = tB + ((uint32_t)((warp & 3) * 32) << 16);  // this warp's lanes
  int cur_mat = -1;
  const bool cosine = (L.flags & NAM_OUT_COSINE) != 0;

  // single material: one copy of the weights for the whole CTA
  if (!MULTI) {
    if (tid == 0 && c_begin < c_end) {
      ptx::fence_proxy_async();
      ptx::mbar_arrive_expect_tx(bar_w, Y.BYTES);
      ptx::bulk_g2s(aW, L.w0, Y.BYTES, bar_w);
      w_pending = true;  // drained by thread 0 at teardown if needed
    }
  }

  constexpr uint32_t ID16 = ptx::idesc_f16(128, 16);
  constexpr uint32_t ID_H = ptx::idesc_f16(128, H);
  constexpr uint32_t ID_N1 = ptx::idesc_f16(128, Y.N1);

  // The thread that issues this chain's MMAs: chain k's in warp k mod 4, so
  // that the issuing warps are spread over the SM's four schedulers.
  auto leader = [&]() -> bool { return ((warp ^ wg) & 3) == 0 && ptx::elect(); };

  // Make this warpgroup's TMEM writes visible to the tensor core, agree on
  // the error state, let one thread issue `issue` and commit it.  False (for
  // every thread of the warpgroup) if a wait of any thread ran out.
  auto stage_issue = [&](auto issue) -> bool {
    ptx::tmem_st_wait();
    ptx::tc_fence_before();
    if (ptx::bar_red_or(bar_id, 128, bad)) {
      bad = true;  // some thread's wait ran out: the whole warpgroup stops
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

  // the leader gives up its weight slot; the barrier before has every thread of
  // the warpgroup done with the slot's weights.  An atomic decrement without
  // the lock: it cannot fail, so no slot stays taken by a warpgroup that has
  // stopped using it.
  auto release_slot = [&]() {
    if (my_slot >= 0) {
      __threadfence_block();
      atomicSub(const_cast<int*>(slot_users + my_slot), 1);
      my_slot = -1;
    }
  };
  int64_t c = c_begin + wg;
  int slot = wg;      // this tile's operand buffer, and the parity of its filling
  uint32_t ph_f = 0;
  TileRef nxt{};
  int64_t i_nxt = 0;  // this row's query in the next tile
  if (c < c_end) {
    nxt = tile_at(L, c);
    if (nxt.count > 0) i_nxt = row_of(nxt);
  }
  for (; c < c_end; c += NCH) {
    const uint32_t bar_full = bar_f + 8 * slot, bar_read = bar_e + 8 * slot, par = ph_f;
    const uint32_t aZ = ptx::smem_u32(smem + S::Z_OFF) + slot * S::ZB;
    slot += NCH;
    if (slot >= NZ) {
      slot -= NZ;
      ph_f ^= 1u;
    }
    const TileRef cur = nxt;
    const int64_t i = i_nxt;
    if (c + NCH < c_end) nxt = tile_at(L, c + NCH);
    if (cur.count <= 0) {
      // an empty slot of a chunk table (count is uniform over the
      // warpgroup): only the hand-over with the fetch warpgroups
      if (c + NCH < c_end && nxt.count > 0) i_nxt = row_of(nxt);
      if (MULTI) {
        if (ptx::bar_red_or(bar_id, 128, bad)) {
          bad = true;
          break;
        }
        if (r == 0) release_slot();  // never held while waiting for an operand
        cur_mat = -1;
      }
      bad |= !ptx::mbar_wait(bar_full, par, L.timeout_ns);
      if (ptx::bar_red_or(bar_id, 128, bad)) {
        bad = true;
        break;
      }
      if (r == 0) ptx::mbar_arrive(bar_read);
      continue;
    }
    const bool valid = r < cur.count;

    // ---- 1. the fetched latent (FP16 halves) -> MMA 1 --------------------
    auto issue1 = [&] {
      ptx::mma_f16(tB + C::D, ptx::sdesc(aZ, 2048, 128), ptx::sdesc(aW + Y.B1, Y.N1 * 16, 128), ID_N1, 0);
      if (FK) ptx::mma_f16(tB + C::F, ptx::sdesc(aConst, 2048, 128), ptx::sdesc(aW + Y.B1B, 256, 128), ID16, 1);
      ptx::mma_commit(bar_read);
    };
    if constexpr (MULTI) {
      // The leader keeps its weight slot only if the tile has the same
      // material and its operand is there already; otherwise it gives the
      // slot up (the barrier: every thread has finished the previous tile),
      // waits for the operand, and then takes a slot holding the material, or
      // loads it into a slot no warpgroup uses (waiting, with the time limit,
      // while all are in use).  A warpgroup that holds a slot therefore never
      // waits for the fetch warpgroups, which may themselves wait for a
      // warpgroup without a slot.
      ptx::tc_fence_before();
      const bool slow = bad || (r == 0 && (cur.mat != cur_mat || !ptx::mbar_test_wait(bar_full, par)));
      if (ptx::bar_red_or(bar_id, 128, slow)) {
        if (r == 0) release_slot();
        bad |= !ptx::mbar_wait(bar_full, par, L.timeout_ns);
        if (r == 0) {
          const uint64_t t0 = ptx::globaltimer();
          int sl = -1, gen = 0;
          bool load = false, ok = !bad && smem_lock(slot_lock, t0, L.timeout_ns);
          while (ok) {
            for (int k = 0; k < S::SLOTS && sl < 0; ++k)
              if (slot_mat[k] == cur.mat) {
                sl = k;
                atomicAdd(const_cast<int*>(slot_users + k), 1);  // (a release takes no lock)
                gen = slot_loads[k];
              }
            for (int k = 0; k < S::SLOTS && sl < 0; ++k)
              if (slot_users[k] == 0) {
                sl = k;
                load = true;
                slot_mat[k] = cur.mat;
                slot_users[k] = 1;
                gen = slot_loads[k] + 1;
                slot_loads[k] = gen;
              }
            smem_unlock(slot_lock);
            if (sl >= 0) break;
            __nanosleep(256);
            // (smem_lock reads the clock only when the lock is taken)
            ok = ptx::globaltimer() - t0 <= L.timeout_ns && smem_lock(slot_lock, t0, L.timeout_ns);
          }
          if (load) {
            const uint32_t bar = bar_w + 8 * sl;
            ptx::fence_proxy_async();
            ptx::mbar_arrive_expect_tx(bar, Y.BYTES);
            ptx::bulk_g2s(ptx::smem_u32(smem + S::W_OFF + sl * S::BLOB_AL), L.mats.weights[cur.mat], Y.BYTES,
                          bar);
          }
          wg_word[wg] = sl >= 0 ? (sl | (gen << 8)) : -1;
          my_slot = sl;
        }
        // broadcast the slot (a failed acquire stops the warpgroup)
        if (ptx::bar_red_or(bar_id, 128, bad)) {
          bad = true;
          break;
        }
        const int word = wg_word[wg];
        if (word < 0) {
          bad = true;
          break;
        }
        const int sl = word & 0xFF, gen = word >> 8;
        aW = ptx::smem_u32(smem + S::W_OFF + sl * S::BLOB_AL);
        bad |= !ptx::mbar_wait(bar_w + 8 * sl, (uint32_t)(gen - 1) & 1u, L.timeout_ns);
        cur_mat = cur.mat;
        if (!stage_issue(issue1)) break;
      } else {
        if (leader()) {
          ptx::tc_fence_after();
          issue1();
          ptx::mma_commit(bar_m);
        }
        mma_pending = true;
      }
    } else {
      if (cur_mat < 0) {
        bad |= !ptx::mbar_wait(bar_w, 0, L.timeout_ns);
        if (!bad && tid == 0) w_pending = false;
        cur_mat = 0;
      }
      bad |= !ptx::mbar_wait(bar_full, par, L.timeout_ns);
      if (!stage_issue(issue1)) break;
    }
    // directions (used after the frame stages) and the masked-pass material,
    // and the next tile's row
    const float wix = ld_field<MULTI>(L.q.wix + i), wiy = ld_field<MULTI>(L.q.wiy + i);
    const float wiz = ld_field<MULTI>(L.q.wiz + i), wox = ld_field<MULTI>(L.q.wox + i);
    const float woy = ld_field<MULTI>(L.q.woy + i), woz = ld_field<MULTI>(L.q.woz + i);
    [[maybe_unused]] const int32_t row_mat = MULTI && L.row_ids ? __ldg(L.row_ids + i) : cur.mat;
    if (c + NCH < c_end && nxt.count > 0) i_nxt = row_of(nxt);
    stage_wait();

    // ---- 2.-3. frame, transformed directions -> MMA 3 -------------------
    float d[12];
    if (FK == 1) {
      {
        uint32_t acc[16];
        ptx::tmem_ld16(tBl + C::F, acc);
        ptx::tmem_ld_wait();
        uint32_t v[16];
#pragma unroll
        for (int j = 0; j < 8; ++j) split_pair<true>(f32_of(acc[2 * j]), f32_of(acc[2 * j + 1]), v[j], v[8 + j]);
        ptx::tmem_st16(tBl + C::A, v);  // (h hi, h lo)
      }
      if (!stage_issue([&] {
            ptx::mma_f16_ts(tB + C::F, tB + C::A, ptx::sdesc(aW + Y.BF2, 256, 128), ID16, 0);
            ptx::mma_f16_ts(tB + C::F, tB + C::A + 8, ptx::sdesc(aW + Y.BF2 + 512, 256, 128), ID16, 1);
          }))
        break;
      stage_wait();
      uint32_t acc[8];
      ptx::tmem_ld8(tBl + C::F, acc);
      ptx::tmem_ld_wait();
      const uint4 b0 = ptx::ld_shared_v4(aW + Y.SB + 32), b1 = ptx::ld_shared_v4(aW + Y.SB + 48);
      const float rr[6] = {f32_of(acc[0]) + f32_of(b0.x), f32_of(acc[1]) + f32_of(b0.y), f32_of(acc[2]) + f32_of(b0.z),
                           f32_of(acc[3]) + f32_of(b0.w), f32_of(acc[4]) + f32_of(b1.x), f32_of(acc[5]) + f32_of(b1.y)};
      const Frame F = build_frame(rr);
      to_local(F, wix, wiy, wiz, d);
      to_local(F, wox, woy, woz, d + 3);
    } else if (FK == 2) {
      uint32_t acc[16];
      ptx::tmem_ld16(tBl + C::F, acc);
      ptx::tmem_ld_wait();
      float rr[12];
#pragma unroll
      for (int j = 0; j < 12; ++j) rr[j] = f32_of(acc[j]);
      const Frame F1 = paper_frame(rr), F2 = paper_frame(rr + 6);
      to_local(F1, wix, wiy, wiz, d);
      to_local(F2, wix, wiy, wiz, d + 3);
      to_local(F1, wox, woy, woz, d + 6);
      to_local(F2, wox, woy, woz, d + 9);
    } else {
      d[0] = wix; d[1] = wiy; d[2] = wiz;
      d[3] = wox; d[4] = woy; d[5] = woz;
    }
    {
      // (d hi, d lo, 1, 0 ...): the 1 meets layer 1's bias column
      if (ND == 6) {
        uint32_t v[8];
        split_pair<false>(d[0], d[1], v[0], v[3]);
        split_pair<false>(d[2], d[3], v[1], v[4]);
        split_pair<false>(d[4], d[5], v[2], v[5]);
        v[6] = 0x00003C00u;
        v[7] = 0u;
        ptx::tmem_st8(tBl + C::A + 8, v);
      } else {
        uint32_t v[16];
#pragma unroll
        for (int j = 0; j < 6; ++j) split_pair<false>(d[2 * j], d[2 * j + 1], v[j], v[6 + j]);
        v[12] = 0x00003C00u;
        v[13] = v[14] = v[15] = 0u;
        ptx::tmem_st16(tBl + C::A, v);
      }
    }
    if (!stage_issue([&] {
          if (ND == 6) {
            ptx::mma_f16_ts(tB + C::D, tB + C::A + 8, ptx::sdesc(aW + Y.BD, H * 16, 128), ID_H, 1);
          } else {
            ptx::mma_f16_ts(tB + C::D, tB + C::A, ptx::sdesc(aW + Y.BD, H * 16, 128), ID_H, 1);
            ptx::mma_f16_ts(tB + C::D, tB + C::A + 8, ptx::sdesc(aW + Y.BD + 2 * H * 16, H * 16, 128), ID_H, 1);
          }
        }))
      break;
    stage_wait();

    // ---- 4. hidden layers: ReLU, FP16 -> next layer ----------------------
    // H = 64: rounded to FP16 once; narrower decoders, where one rounded
    // layer already takes a large share of the FP16 error budget, keep (hi,
    // lo) halves here too (lo in the operand columns [H + 16, H + 16 + H/2)).
    // FP8 (P8): each hidden -> hidden layer has E4M3 weights (codes of
    // W / s_w); its input x enters as two E4M3 code sets of x / s_a, hi =
    // E4M3(x / s_a) and lo = E4M3(x / s_a - hi), in [H, H + H/4) and
    // [H + H/4, H + H/2) (four codes per column), so that the accumulator
    // holds sum (hi + lo) code_w = (pre-activation - b) / c, c = s_a s_w; the
    // next epilogue restores c D + b in FP32.
    constexpr bool SPLIT_HID = H < 64 && !P8;
    constexpr int NC = 16;
    constexpr uint32_t ID8_H = ptx::idesc_e4m3(128, H);
    bool ok = true;
    // (multiplier, bias) that turn the accumulator into the pre-activation
    // of the layer that wrote it: (1, 0) after an FP16 layer (bias in the MMA)
    float pre_c = 1.0f;
    uint32_t pre_b = 0;  // shared-memory address of the FP32 bias, 0: none
#pragma unroll
    for (int layer = 0; layer < NH - 1; ++layer) {
      const int boff = Y.BH + layer * H * (H + 16) * 2;
      if constexpr (P8) {
        const float inv_sa = reinterpret_cast<const float*>(smem + (aW - aConst) + Y.SB)[2 * layer];
#pragma unroll
        for (int c0 = 0; c0 < H; c0 += 16) {
          uint32_t acc[16];
          ptx::tmem_ld16(tBl + C::D + c0, acc);
          ptx::tmem_ld_wait();
          float t[16];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint4 b = pre_b ? ptx::ld_shared_v4(pre_b + 4 * (c0 + 4 * q)) : make_uint4(0u, 0u, 0u, 0u);
            const float2 t01 = ptx::fma2(make_float2(f32_of(acc[4 * q]), f32_of(acc[4 * q + 1])),
                                         make_float2(pre_c, pre_c), make_float2(f32_of(b.x), f32_of(b.y)));
            const float2 t23 = ptx::fma2(make_float2(f32_of(acc[4 * q + 2]), f32_of(acc[4 * q + 3])),
                                         make_float2(pre_c, pre_c), make_float2(f32_of(b.z), f32_of(b.w)));
            t[4 * q] = fmaxf(t01.x, 0.0f) * inv_sa;
            t[4 * q + 1] = fmaxf(t01.y, 0.0f) * inv_sa;
            t[4 * q + 2] = fmaxf(t23.x, 0.0f) * inv_sa;
            t[4 * q + 3] = fmaxf(t23.y, 0.0f) * inv_sa;
          }
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t h2[2], l2[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float x0 = t[4 * q + 2 * e], x1 = t[4 * q + 2 * e + 1];
              h2[e] = ptx::pack_e4m3x2(x0, x1);
              const float2 hv = ptx::unpack_e4m3x2(h2[e]);
              const float2 d = ptx::sub2(make_float2(x0, x1), hv);
              l2[e] = ptx::pack_e4m3x2(d.x, d.y);
            }
            hi[q] = h2[0] | (h2[1] << 16);
            lo[q] = l2[0] | (l2[1] << 16);
          }
          ptx::tmem_st4(tBl + C::HID + c0 / 4, hi);
          ptx::tmem_st4(tBl + C::HID + H / 4 + c0 / 4, lo);
        }
        if (!stage_issue([&] {
#pragma unroll
              for (int s = 0; s < (2 * H) / 32; ++s)
                ptx::mma_f8_ts(tB + C::D, tB + C::HID + 8 * s, ptx::sdesc(aW + boff + s * 2 * H * 16, H * 16, 128),
                               ID8_H, s > 0 ? 1u : 0u);
            })) {
          ok = false;
          break;
        }
        pre_c = reinterpret_cast<const float*>(smem + (aW - aConst) + Y.SB)[2 * layer + 1];
        pre_b = aW + boff + 2 * H * H;
      } else if constexpr (SPLIT_HID) {
#pragma unroll
        for (int c0 = 0; c0 < H; c0 += 16) {
          uint32_t acc[16];
          ptx::tmem_ld16(tBl + C::D + c0, acc);
          ptx::tmem_ld_wait();
          uint32_t hi[8], lo[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) split_pair<true>(f32_of(acc[2 * j]), f32_of(acc[2 * j + 1]), hi[j], lo[j]);
          ptx::tmem_st8(tBl + C::HID + c0 / 2, hi);
          ptx::tmem_st8(tBl + C::A + c0 / 2, lo);
        }
      } else {
#pragma unroll
        for (int c0 = 0; c0 < H; c0 += NC) {
          uint32_t acc[NC];
          ptx::tmem_ld16(tBl + C::D + c0, acc);
          ptx::tmem_ld_wait();
          uint32_t pk[NC / 2];
#pragma unroll
          for (int j = 0; j < NC / 2; ++j) pk[j] = ptx::pack_h2_relu(f32_of(acc[2 * j]), f32_of(acc[2 * j + 1]));
          ptx::tmem_st8(tBl + C::HID + c0 / 2, pk);
        }
      }
      if constexpr (!P8) {
        if (!stage_issue([&] {
#pragma unroll
              for (int s = 0; s < H / 16; ++s)
                ptx::mma_f16_ts(tB + C::D, tB + C::HID + 8 * s, ptx::sdesc(aW + boff + s * 2 * H * 16, H * 16, 128),
                                ID_H, s > 0 ? 1u : 0u);
              if constexpr (SPLIT_HID) {
#pragma unroll
                for (int s = 0; s < H / 16; ++s)
                  ptx::mma_f16_ts(tB + C::D, tB + C::A + 8 * s, ptx::sdesc(aW + boff + s * 2 * H * 16, H * 16, 128),
                                  ID_H, 1u);
              }
              ptx::mma_f16(tB + C::D, ptx::sdesc(aConst, 2048, 128),
                           ptx::sdesc(aW + boff + (H / 8) * H * 16, H * 16, 128), ID_H, 1u);
            })) {
          ok = false;
          break;
        }
      }
      stage_wait();
    }
    if (!ok) break;

    // ---- 5. output layer -----------------------------------------------------
    float y[6];  // RGB, then (albedo head) the albedo
    const bool alb = L.albedo != nullptr;
    {
      // in FP32 on the last hidden layer (even and odd units as the halves of
      // packed FMAs); weights from the kernel's parameters, or, when the
      // launch mixes materials, from shared memory: the same operations in the
      // same order
      float2 s[6];
#pragma unroll
      for (int o = 0; o < 6; ++o) {
        if constexpr (MULTI) s[o] = make_float2(ptx::ld_shared_f1(aW + Y.SB + 64 + 4 * o), 0.0f);
        else s[o] = make_float2(O.bo[o], 0.0f);
      }
#pragma unroll
      for (int c0 = 0; c0 < H; c0 += 16) {
        uint32_t acc[16];
        ptx::tmem_ld16(tBl + C::D + c0, acc);
        ptx::tmem_ld_wait();
        float h[16];
        if constexpr (P8) {
          // the last hidden layer was an E4M3 layer: pre-activation = c D + b
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint4 b = ptx::ld_shared_v4(pre_b + 4 * (c0 + 4 * q));
            const float2 t01 = ptx::fma2(make_float2(f32_of(acc[4 * q]), f32_of(acc[4 * q + 1])),
                                         make_float2(pre_c, pre_c), make_float2(f32_of(b.x), f32_of(b.y)));
            const float2 t23 = ptx::fma2(make_float2(f32_of(acc[4 * q + 2]), f32_of(acc[4 * q + 3])),
                                         make_float2(pre_c, pre_c), make_float2(f32_of(b.z), f32_of(b.w)));
            acc[4 * q] = __float_as_uint(t01.x);
            acc[4 * q + 1] = __float_as_uint(t01.y);
            acc[4 * q + 2] = __float_as_uint(t23.x);
            acc[4 * q + 3] = __float_as_uint(t23.y);
          }
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float a = f32_of(acc[k]);
          h[k] = a + fabsf(a);
        }
        auto dot = [&](int o) {
#pragma unroll
          for (int k = 0; k < 16; k += 4) {
            float4 w;
            if constexpr (MULTI) {
              const uint4 v = ptx::ld_shared_v4(aW + Y.WO + 4 * (o * H + c0 + k));
              w = make_float4(f32_of(v.x), f32_of(v.y), f32_of(v.z), f32_of(v.w));
            } else {
              w = make_float4(O.wo[o][c0 + k], O.wo[o][c0 + k + 1], O.wo[o][c0 + k + 2], O.wo[o][c0 + k + 3]);
            }
            s[o] = ptx::fma2(make_float2(w.x, w.y), make_float2(h[k], h[k + 1]), s[o]);
            s[o] = ptx::fma2(make_float2(w.z, w.w), make_float2(h[k + 2], h[k + 3]), s[o]);
          }
        };
#pragma unroll
        for (int o = 0; o < 3; ++o) dot(o);
        if (alb) {
#pragma unroll
          for (int o = 3; o < 6; ++o) dot(o);
        }
      }
#pragma unroll
      for (int o = 0; o < 6; ++o) y[o] = s[o].x + s[o].y;
    }

    // ---- output ---------------------------------------------------------------
    if (valid && (!MULTI || row_mat == cur.mat)) {
      if (alb) {
        // no cosine factor on the albedo
        L.albedo[3 * i + 0] = y[3];
        L.albedo[3 * i + 1] = y[4];
        L.albedo[3 * i + 2] = y[5];
      }
      const float cz = cosine ? fmaxf(wiz, 0.0f) : 1.0f;
      L.rgb[3 * i + 0] = y[0] * cz;
      L.rgb[3 * i + 1] = y[1] * cz;
      L.rgb[3 * i + 2] = y[2] * cz;
    }
    ptx::tc_fence_before();
  }
  if constexpr (MULTI) {
    // every thread is past its last reads of the slot's weights (the output
    // layer takes them from shared memory) before another chain may load over
    // them; all threads of a warpgroup leave the loop together
    ptx::bar_sync(bar_id, 128);
    if (r == 0) release_slot();
  }
  }  // chain warpgroups

  // ---- teardown -------------------------------------------------------------
  // MMAs and bulk copies still in flight after a wait gave up are waited for
  // with the fixed drain limit, and TMEM is freed only if they all completed.
  bool drained = true;
  if (r == 0 && mma_pending) drained &= ptx::mbar_wait(bar0 + 8 * wg, ph_m ^ 1, ptx::kDrainTimeoutNs);
  if (!MULTI && tid == 0 && w_pending) drained &= ptx::mbar_wait(bar_w, 0, ptx::kDrainTimeoutNs);
  if (MULTI) {
    __syncthreads();  // every warpgroup has left its loop: no slot is loaded after this
    if (tid == 0)
      for (int k = 0; k < S::SLOTS; ++k)
        if (slot_loads[k] > 0)
          drained &= ptx::mbar_wait(bar_w + 8 * k, (uint32_t)(slot_loads[k] - 1) & 1u, ptx::kDrainTimeoutNs);
  }
  if (bad) record_error(L.err, DEVERR_WAIT_TIMEOUT);
  if (!drained) record_error(L.err, DEVERR_DRAIN_TIMEOUT);
  ptx::tc_fence_before();
  const bool all_drained = __syncthreads_and(drained ? 1 : 0) != 0;
  if (warp == 0 && all_drained) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(*tslot, 512);
  }
}

// ---------------------------------------------------------------------------
// host launch
// ---------------------------------------------------------------------------
// One material: five chains (TMEM 5 x (H + 32) <= 480 of 512 columns) and two
// fetch warpgroups, 896 threads at <= 72 registers (1920x1080, H = 64: 90 us;
// three fetch warpgroups at 64 registers 96, four chains 97).  Four and three
// where the fetch is the longer side: mixed materials, whose fetch also follows
// the binning permutation (a material per pixel at 1920x1080: 250 us; 5 + 2
// 263, 5 + 3 277); FP32 texels, two loads and sectors of HBM traffic each
// (1.5 M queries, 2048^2, H = 16 .. 64: 81 .. 105 us, 5 + 2 95 .. 124; not FP8
// with three hidden layers, 126 against 120); and H = 16 in FP16, whose chains
// are short (52 .. 64 us, 5 + 2 60 .. 74; H = 32 with a frame 70 against 66).
template <int H, int FK, int NH, bool F16P, bool MULTI, bool P8>
static int launch_f16_one(const LaunchCommon& L, cudaStream_t s) {
  constexpr bool kFetch3 = MULTI || (F16P ? H == 16 && !P8 : !(P8 && NH == 3));
  constexpr int NCH = kFetch3 ? 4 : 5, NF = kFetch3 ? 3 : 2;
  using S = F16Smem<H, FK, NH, F16P, MULTI, NCH, NF>;
  static_assert(S::BYTES <= 227 * 1024, "shared memory");
  static_assert(NCH * F16Cols<H>::COLS <= 512, "TMEM columns");
  auto k = eval_f16_kernel<H, FK, NH, F16P, MULTI, NCH, NF, P8>;
  static std::atomic<uint64_t> configured{0};
  once_per_device(configured, [&] {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, S::BYTES);
    // the smallest carveout that holds the CTA: the rest of the SM's
    // L1/shared storage caches the texel gathers
    const int pct = (S::BYTES + 1024) * 100 / (228 * 1024) + 1;
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
  });
  const int64_t ntiles = L.chunks ? (int64_t)L.n_chunks : (L.n + 127) / 128;
  if (ntiles == 0) return 0;
  // a small launch spreads its tiles over the SMs
  const int grid = (int)(ntiles < L.num_sms ? ntiles : L.num_sms);
  OutParams<H, MULTI> O;
  if constexpr (!MULTI) {
    for (int o = 0; o < 6; ++o) {
      std::memcpy(O.wo[o], L.nw->wo[o], sizeof O.wo[o]);
      O.bo[o] = L.nw->bo[o];
    }
  }
  k<<<grid, (NCH + NF) * 128, S::BYTES, s>>>(L, O);
  return (int)cudaGetLastError();
}

template <int H, int FK, int NH, bool P8>
static int f16_pick(const LaunchCommon& L, cudaStream_t s) {
  const bool f16 = L.pyr.f16 != 0, multi = L.chunks != nullptr;
  if (f16)
    return multi ? launch_f16_one<H, FK, NH, true, true, P8>(L, s) : launch_f16_one<H, FK, NH, true, false, P8>(L, s);
  return multi ? launch_f16_one<H, FK, NH, false, true, P8>(L, s) : launch_f16_one<H, FK, NH, false, false, P8>(L, s);
}

template <int H, int NH, bool P8>
static int f16_frame(const LaunchCommon& L, cudaStream_t s) {
  switch (L.shape.frame) {
    case 0: return f16_pick<H, 0, NH, P8>(L, s);
    case 1: return f16_pick<H, 1, NH, P8>(L, s);
    case 2: return f16_pick<H, 2, NH, P8>(L, s);
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace nam
