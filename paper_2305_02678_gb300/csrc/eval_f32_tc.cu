// FP32 evaluation on the tensor cores, for materials whose weights do not
// change (a trainable material's masters may be written between launches: it
// keeps the per-thread kernel of fwd_f32.cu).
//
// Rows whose decoder input is not finite, or so large that a layer could
// overflow (a bound from the weights' norms), are evaluated per thread.
//
// Latent filter, frame MLP, frame build, direction transform and output layer
// run in FP32 per thread, in the per-thread kernel's order of operations; the
// decoder's wide layers run as bf16 MMAs on three-way splits: an activation
// x = x_h + x_m + x_l (each the next 8 significant bits, cut off, so the sum
// is x itself) and a weight W = W_h + W_m + W_l (each rounded to nearest).
// The six products down to 2^-16 relative are accumulated in FP32; what is
// left out is below 1.5 2^-23 of a term and of either sign.  bf16 has FP32's exponent range, so
// nothing is scaled.  The tensor core's accumulator cuts off instead of
// rounding, once per MMA (K = 16), so the small products come first, then the
// bias, then the leading product's few MMAs (with the bias first the error
// against 64 bits was 1.2 to 2.5 times the per-thread kernel's).
// Error against 64 bits, norm of the difference over norm of the result, as a
// multiple of the per-thread kernel's (30,000 queries, four seeds; Glorot,
// positive, heavy-tailed, sparse, scaled weights, large biases): H = 64 0.40 ..
// 0.97, H = 32 0.42 .. 1.07, H = 16 0.47 .. 1.07.
//
// Structure as in eval_tc.cuh: fetch warpgroups filter the latents, a chain
// warpgroup takes a tile of 128 queries through the layers, two (or three)
// MMA round trips per tile.  TMEM columns of a chain: accumulator [0, H),
// then the operand: three terms of the decoder input (KX / 2 columns each)
// or of a hidden layer (H / 2 columns each).
// What bounds it: at H = 64, three chains per SM (160 columns each): 20 warps
// keep 57 % of the issue slots (the splits take 11 instructions per pair of
// activations) and 35 % of the tensor pipe busy.
// 1280x720, H = 64, frame MLP: 81 us, 334 in the per-thread kernel (fed from
// shared memory at a third of the FP32 rate).
#include "eval_tc.cuh"
#include "f32_body.cuh"

namespace nam {
namespace {

// weight blob: MMA B operands, canonical no-swizzle K-major, bf16
struct F32Lay {
  int KX;    // K of the first layer: decoder inputs, then 1 (meets the bias), zero padding: 16, or 32 (paper frame)
  int B1;    // 3 blocks (h, m, l) of H x KX
  int BH;    // per hidden -> hidden layer: 3 blocks of H x H, then H x 16: the bias terms in columns 0..2
  int BYTES;
};
__host__ __device__ constexpr F32Lay f32_lay(int H, int FK, int NH) {
  F32Lay o{};
  o.KX = FK == 2 ? 32 : 16;
  o.B1 = 0;
  o.BH = 3 * H * o.KX * 2;
  o.BYTES = o.BH + (NH - 1) * (3 * H * H + 16 * H) * 2;
  return o;
}

// FP32 layers that run per thread; weights as constant-bank operands
template <int H>
struct F32Params {
  float f1[8][16], fb1[16];  // frame layer 1, [input][unit] (paper form: 12 units, its only layer)
  float f2[6][16], fb2[6];   // frame MLP layer 2, [output][input]
  float wo[6][H], bo[6];     // output layer
  float n2_max;              // |x|^2 up to which no layer can overflow
};

template <int H, int FK, int NH, int NCH, int NF>
struct F32Smem {
  static constexpr F32Lay Y = f32_lay(H, FK, NH);
  static constexpr int W_OFF = 4096;  // after the constant block (ones in columns 0..2) and the zero block
  static constexpr int Z_OFF = W_OFF + (Y.BYTES + 127) / 128 * 128;
  static constexpr int ZB = 4096;  // z of 128 rows, FP32, two 16-byte halves
  static constexpr int NZ = NCH % NF ? NCH * NF : NCH;  // as F16Smem::NZ
  static constexpr int BAR_OFF = Z_OFF + NZ * ZB;
  static constexpr int TSLOT_OFF = (BAR_OFF + 8 * (NCH + 2 * NZ + 1) + 15) / 16 * 16;
  static constexpr int BYTES = TSLOT_OFF + 16;
};

// dot_row with the weights anywhere in memory: the same two sums
template <int N>
__device__ __forceinline__ float dot_row_any(const float* __restrict__ row, const float* h) {
  float s0 = 0.0f, s1 = 0.0f;
#pragma unroll 4
  for (int k = 0; k < N; k += 2) {
    s0 = fmaf(row[k], h[k], s0);
    s1 = fmaf(row[k + 1], h[k + 1], s1);
  }
  return s0 + s1;
}

// One query with the weights in global memory, for the rows of which a split
// might not be finite (an infinity has none: its lower terms are NaN), because
// their inputs are not or because a layer could overflow.  The operations of
// eval_query in its order: the per-thread kernel's results bit for bit.
template <int H, int NH, int FK, bool F16P>
__device__ __noinline__ void eval_slow(const LaunchCommon& L, int64_t i, float y[6]) {
  const float* p = L.masters;
  float z[8], x[20];
  fetch_latent<F16P>(L.pyr, L.pyr0, L.q.u[i], L.q.v[i], L.q.lod[i], L.q.xi ? L.q.xi[i] : 0.0f, z);
  const float wi[3] = {L.q.wix[i], L.q.wiy[i], L.q.wiz[i]}, wo[3] = {L.q.wox[i], L.q.woy[i], L.q.woz[i]};
  for (int c = 0; c < 8; ++c) x[c] = z[c];
  constexpr int IN = FK == 2 ? 20 : 14;
  // the frame layer on z: its unit j
  auto unit = [&](int j, int bias) {
    float s = p[bias + j];
    for (int c = 0; c < 8; ++c) s = fmaf(p[j * 8 + c], z[c], s);
    return s;
  };
  if (FK == 1) {
    float hf[16], r[6];
    for (int j = 0; j < 16; ++j) hf[j] = fmaxf(unit(j, 128), 0.0f);
    for (int j = 0; j < 6; ++j) r[j] = p[240 + j] + dot_row_any<16>(p + 144 + j * 16, hf);
    const Frame F = build_frame(r);
    to_local(F, wi[0], wi[1], wi[2], x + 8);
    to_local(F, wo[0], wo[1], wo[2], x + 11);
    p += 246;
  } else if (FK == 2) {
    float r[12];
    for (int j = 0; j < 12; ++j) r[j] = unit(j, 96);
    const Frame F1 = paper_frame(r), F2 = paper_frame(r + 6);
    to_local(F1, wi[0], wi[1], wi[2], x + 8);
    to_local(F2, wi[0], wi[1], wi[2], x + 11);
    to_local(F1, wo[0], wo[1], wo[2], x + 14);
    to_local(F2, wo[0], wo[1], wo[2], x + 17);
    p += 108;
  } else {
    for (int c = 0; c < 3; ++c) {
      x[8 + c] = wi[c];
      x[11 + c] = wo[c];
    }
  }
  float a[H], b[H];
  for (int j = 0; j < H; ++j) a[j] = fmaxf(p[IN * H + j] + dot_row_any<IN>(p + j * IN, x), 0.0f);
  p += IN * H + H;
  for (int l = 1; l < NH; ++l) {
    for (int j = 0; j < H; ++j) b[j] = fmaxf(p[H * H + j] + dot_row_any<H>(p + j * H, a), 0.0f);
    for (int j = 0; j < H; ++j) a[j] = b[j];
    p += H * H + H;
  }
  for (int o = 0; o < L.shape.out; ++o) {
    float s = p[L.shape.out * H + o];
    for (int k = 0; k < H; ++k) s = fmaf(p[o * H + k], a[k], s);
    y[o] = s;
  }
}

template <int H, int FK, int NH, bool F16P, int NCH, int NF>
__global__ void __launch_bounds__((NCH + NF) * 128, 1)
    eval_f32_tc_kernel(const __grid_constant__ LaunchCommon L, const __grid_constant__ F32Params<H> O) {
  using S = F32Smem<H, FK, NH, NCH, NF>;
  constexpr F32Lay Y = S::Y;
  constexpr int NZ = S::NZ, KX = Y.KX;
  constexpr int XC = 3 * (KX > H ? KX : H) / 2;  // operand columns
  constexpr int COLS = H + XC;
  static_assert(NCH * COLS <= 512, "TMEM columns");
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, r = tid & 127;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0), wg = warp >> 2;
  const uint32_t aConst = ptx::smem_u32(smem), aW = ptx::smem_u32(smem + S::W_OFF);
  const uint32_t bar0 = ptx::smem_u32(smem + S::BAR_OFF);
  const uint32_t bar_f = bar0 + 8 * NCH, bar_e = bar0 + 8 * (NCH + NZ), bar_w = bar0 + 8 * (NCH + 2 * NZ);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + S::TSLOT_OFF);
  if (tid == 0) {
    for (int k = 0; k < NCH; ++k) ptx::mbar_init(bar0 + 8 * k, 1);
    for (int k = 0; k < NZ; ++k) {
      ptx::mbar_init(bar_f + 8 * k, 4);  // the four warps of a fetch warpgroup
      ptx::mbar_init(bar_e + 8 * k, 4);  // the four warps of a chain
    }
    ptx::mbar_init(bar_w, 1);
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_u32(tslot), 512);
    ptx::tmem_relinquish();
  }
  if (tid < 128) {
    ptx::st_shared_v4(aConst + tid * 16, 0x3F803F80u, 0x00003F80u, 0u, 0u);
    ptx::st_shared_v4(aConst + 2048 + tid * 16, 0u, 0u, 0u, 0u);
  }
  ptx::fence_proxy_async();
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
    bad = !fetch_loop<F16P, false, true, NF, NZ>(
        L, c_begin, c_end, wg - NCH, bar_f, bar_e, bad,
        [&](const TileRef&) { return reinterpret_cast<const uint8_t*>(L.pyr0); }, row_of,
        [](const TileRef&) {}, [&](int slot, const float z[8]) {
          const uint32_t zs = ptx::smem_u32(smem + S::Z_OFF) + slot * S::ZB + r * 16;
          auto u = [](float v) { return __float_as_uint(v); };
          ptx::st_shared_v4(zs, u(z[0]), u(z[1]), u(z[2]), u(z[3]));
          ptx::st_shared_v4(zs + 2048, u(z[4]), u(z[5]), u(z[6]), u(z[7]));
        });
  } else {
    const uint32_t bar_m = bar0 + 8 * wg, bar_id = 1 + wg;
    const uint32_t tD = tmem + wg * COLS, tX = tD + H;       // MMA addresses (lane 0)
    const uint32_t lane = (uint32_t)((warp & 3) * 32) << 16;  // this warp's lanes
    const bool cosine = (L.flags & NAM_OUT_COSINE) != 0, alb = L.albedo != nullptr;
    if (tid == 0 && c_begin < c_end) {
      ptx::fence_proxy_async();
      ptx::mbar_arrive_expect_tx(bar_w, Y.BYTES);
      ptx::bulk_g2s(aW, L.w0, Y.BYTES, bar_w);
      w_pending = true;
    }
    constexpr uint32_t ID = ptx::idesc_bf16(128, H);
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
    // D = the six products of the operand terms (h, m, l of K columns in
    // all, at tX) with the weight blocks at b; small products first (an
    // accumulator at full magnitude would cut each of them off at its last
    // bit), then `bias`, then the leading product
    auto products = [&](uint32_t b, int K, auto bias) {
      const int kc = K / 2;                       // columns of a term
      const uint32_t blk = (uint32_t)H * K * 2;   // bytes of a weight block
      const int at[6] = {2, 1, 0, 1, 0, 0};       // operand term (h, m, l = 0, 1, 2)
      const int bt[6] = {0, 1, 2, 0, 1, 0};       // weight term
#pragma unroll
      for (int t = 0; t < 6; ++t) {
        if (t == 5) bias();
#pragma unroll
        for (int s = 0; s < K / 16; ++s)
          ptx::mma_f16_ts(tD, tX + at[t] * kc + 8 * s, ptx::sdesc(b + bt[t] * blk + s * 2 * H * 16, H * 16, 128), ID,
                          t + s > 0 ? 1u : 0u);
      }
    };

    int slot = wg;
    uint32_t ph_f = 0;
    bool w_ready = false;
    for (int64_t c = c_begin + wg; c < c_end; c += NCH) {
      const TileRef cur = tile_at(L, c);
      const bool valid = r < cur.count;
      const int64_t i = row_of(cur);
      const float wix = ld_field<false>(L.q.wix + i), wiy = ld_field<false>(L.q.wiy + i);
      const float wiz = ld_field<false>(L.q.wiz + i), wox = ld_field<false>(L.q.wox + i);
      const float woy = ld_field<false>(L.q.woy + i), woz = ld_field<false>(L.q.woz + i);
      if (!w_ready) {
        bad |= !ptx::mbar_wait(bar_w, 0, L.timeout_ns);
        if (!bad && tid == 0) w_pending = false;
        w_ready = true;
      }
      // ---- decoder input x = (z, T wi, T wo, 1) ------------------------------
      bad |= !ptx::mbar_wait(bar_f + 8 * slot, ph_f, L.timeout_ns);
      float x[KX];
      {
        const uint32_t zs = ptx::smem_u32(smem + S::Z_OFF) + slot * S::ZB + r * 16;
        const uint4 z0 = ptx::ld_shared_v4(zs), z1 = ptx::ld_shared_v4(zs + 2048);
        x[0] = f32_of(z0.x); x[1] = f32_of(z0.y); x[2] = f32_of(z0.z); x[3] = f32_of(z0.w);
        x[4] = f32_of(z1.x); x[5] = f32_of(z1.y); x[6] = f32_of(z1.z); x[7] = f32_of(z1.w);
      }
      __syncwarp();
      if ((tid & 31) == 0) ptx::mbar_arrive(bar_e + 8 * slot);
      slot += NCH;
      if (slot >= NZ) {
        slot -= NZ;
        ph_f ^= 1u;
      }
      if constexpr (FK == 1) {
        float2 h[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          h[j] = make_float2(O.fb1[2 * j], O.fb1[2 * j + 1]);
#pragma unroll
          for (int k = 0; k < 8; ++k)
            h[j] = ptx::fma2(make_float2(O.f1[k][2 * j], O.f1[k][2 * j + 1]), make_float2(x[k], x[k]), h[j]);
          h[j].x = fmaxf(h[j].x, 0.0f);
          h[j].y = fmaxf(h[j].y, 0.0f);
        }
        float rr[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          float2 s = make_float2(0.0f, 0.0f);  // even and odd inputs
#pragma unroll
          for (int k = 0; k < 8; ++k)
            s = ptx::fma2(make_float2(O.f2[j][2 * k], O.f2[j][2 * k + 1]), h[k], s);
          rr[j] = O.fb2[j] + (s.x + s.y);
        }
        const Frame F = build_frame(rr);
        to_local(F, wix, wiy, wiz, x + 8);
        to_local(F, wox, woy, woz, x + 11);
      } else if constexpr (FK == 2) {
        float rr[12];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          float2 s = make_float2(O.fb1[2 * j], O.fb1[2 * j + 1]);
#pragma unroll
          for (int k = 0; k < 8; ++k)
            s = ptx::fma2(make_float2(O.f1[k][2 * j], O.f1[k][2 * j + 1]), make_float2(x[k], x[k]), s);
          rr[2 * j] = s.x;
          rr[2 * j + 1] = s.y;
        }
        const Frame F1 = paper_frame(rr), F2 = paper_frame(rr + 6);
        to_local(F1, wix, wiy, wiz, x + 8);
        to_local(F2, wix, wiy, wiz, x + 11);
        to_local(F1, wox, woy, woz, x + 14);
        to_local(F2, wox, woy, woz, x + 17);
      } else {
        x[8] = wix; x[9] = wiy; x[10] = wiz;
        x[11] = wox; x[12] = woy; x[13] = woz;
      }
      constexpr int IN = FK == 2 ? 20 : 14;
      x[IN] = 1.0f;
#pragma unroll
      for (int k = IN + 1; k < KX; ++k) x[k] = 0.0f;
      float2 n2 = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int k = 0; k < KX; k += 2) n2 = ptx::fma2(make_float2(x[k], x[k + 1]), make_float2(x[k], x[k + 1]), n2);
      // an infinity or NaN in z or a direction makes it through the frame to x
      const bool in_range = n2.x + n2.y <= O.n2_max;
#pragma unroll
      for (int k0 = 0; k0 < KX; k0 += 16) {
        uint32_t h[8], m[8], l[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) ptx::split3(x[k0 + 2 * j], x[k0 + 2 * j + 1], h[j], m[j], l[j]);
        ptx::tmem_st8(tX + lane + k0 / 2, h);
        ptx::tmem_st8(tX + lane + KX / 2 + k0 / 2, m);
        ptx::tmem_st8(tX + lane + KX + k0 / 2, l);
      }
      if (!stage_issue([&] { products(aW + Y.B1, KX, [] {}); })) break;
      stage_wait();
      // ---- hidden layers ------------------------------------------------------
      bool ok = true;
#pragma unroll
      for (int layer = 0; layer < NH - 1; ++layer) {
        const uint32_t b = aW + Y.BH + layer * (3 * H * H + 16 * H) * 2;
#pragma unroll
        for (int c0 = 0; c0 < H; c0 += 16) {
          uint32_t acc[16];
          ptx::tmem_ld16(tD + lane + c0, acc);
          ptx::tmem_ld_wait();
          uint32_t h[8], m[8], l[8];
#pragma unroll
          for (int j = 0; j < 8; ++j)
            ptx::split3(fmaxf(f32_of(acc[2 * j]), 0.0f), fmaxf(f32_of(acc[2 * j + 1]), 0.0f), h[j], m[j], l[j]);
          ptx::tmem_st8(tX + lane + c0 / 2, h);
          ptx::tmem_st8(tX + lane + H / 2 + c0 / 2, m);
          ptx::tmem_st8(tX + lane + H + c0 / 2, l);
        }
        if (!stage_issue([&] {
              products(b, H, [&] {
                // its terms on the constant block
                ptx::mma_f16(tD, ptx::sdesc(aConst, 2048, 128), ptx::sdesc(b + 3 * H * H * 2, H * 16, 128), ID, 1u);
              });
            })) {
          ok = false;
          break;
        }
        stage_wait();
      }
      if (!ok) break;
      // ---- output layer ---------------------------------------------------------
      float2 s[6];
#pragma unroll
      for (int o = 0; o < 6; ++o) s[o] = make_float2(O.bo[o], 0.0f);
#pragma unroll
      for (int c0 = 0; c0 < H; c0 += 16) {
        uint32_t acc[16];
        ptx::tmem_ld16(tD + lane + c0, acc);
        ptx::tmem_ld_wait();
        float h[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) h[k] = fmaxf(f32_of(acc[k]), 0.0f);
        // sixteen units at a time, so that no partial sum takes more than
        // a dozen roundings
        auto dot = [&](int o) {
          float2 t = make_float2(0.0f, 0.0f);
#pragma unroll
          for (int k = 0; k < 16; k += 2)
            t = ptx::fma2(make_float2(O.wo[o][c0 + k], O.wo[o][c0 + k + 1]), make_float2(h[k], h[k + 1]), t);
          s[o].x += t.x;
          s[o].y += t.y;
        };
#pragma unroll
        for (int o = 0; o < 3; ++o) dot(o);
        if (alb) {
#pragma unroll
          for (int o = 3; o < 6; ++o) dot(o);
        }
      }
      float y[6];
#pragma unroll
      for (int o = 0; o < 6; ++o) y[o] = s[o].x + s[o].y;
      if (valid) {
        if (!in_range) eval_slow<H, NH, FK, F16P>(L, i, y);
        if (alb) {
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
  }

  // ---- teardown (as in eval_tc.cuh) ------------------------------------------
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

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------
// bf16 of x, round to nearest even; the bits
uint16_t bf16_rn(float x) {
  uint32_t b;
  std::memcpy(&b, &x, 4);
  return (uint16_t)((b + 0x7FFFu + ((b >> 16) & 1u)) >> 16);
}
float bf16_val(uint16_t h) {
  const uint32_t b = (uint32_t)h << 16;
  float f;
  std::memcpy(&f, &b, 4);
  return f;
}
// w (1 + kCut) = h + m + l, each rounded to nearest; false if h overflows.
// kCut: the accumulator cuts off towards zero, on average 4e-8 of the value
// per layer (measured: the mean signed error against 64 bits of every shape was
// that much per layer; with it compensated here, below 5e-8 for a whole decoder
// of any of the families of weights above)
constexpr double kCut = 4e-8;
bool bf16_split(float w, uint16_t t[3]) {
  double x = (double)w * (1.0 + kCut);
  for (int k = 0; k < 3; ++k) {
    t[k] = bf16_rn((float)x);
    const float v = bf16_val(t[k]);
    if (!std::isfinite(v)) return false;
    x -= v;
  }
  return true;
}

// The largest |x|^2 of a decoder input x (with the 1 that meets the bias) for
// which every product, partial sum and activation of every layer stays below
// 2^120: |h_l| <= |W_l| |h_{l-1}| + |b_l| in Euclidean and Frobenius norms,
// followed through the layers as a |x| + c.  `dec`: n layers, widths w[0 .. n].
double input_limit(const float* dec, const int* w, int n) {
  const double top = 0x1p120;
  auto norm = [](const float* p, int k) {
    double s = 0.0;
    for (int i = 0; i < k; ++i) s += (double)p[i] * p[i];
    return std::sqrt(s);
  };
  double a = 1.0, c = 0.0, r = 0x1p64;
  for (int l = 0; l < n; ++l) {
    const int nw = w[l + 1] * w[l];
    const double fw = norm(dec, nw), fb = norm(dec + nw, w[l + 1]);
    a *= l == 0 ? std::hypot(fw, fb) : fw;
    c = l == 0 ? 0.0 : fw * c + fb;
    r = std::fmin(r, (top - c) / std::fmax(a, 1e-300));
    dec += nw + w[l + 1];
  }
  return r < 0.0 ? 0.0 : r * r;
}

template <int H>
F32Params<H> f32_params(const NarrowW& n) {
  F32Params<H> O;
  std::memcpy(O.f1, n.f1, sizeof O.f1);
  std::memcpy(O.fb1, n.fb1, sizeof O.fb1);
  std::memcpy(O.f2, n.f2, sizeof O.f2);
  std::memcpy(O.fb2, n.fb2, sizeof O.fb2);
  for (int o = 0; o < 6; ++o) std::memcpy(O.wo[o], n.wo[o], sizeof O.wo[o]);
  std::memcpy(O.bo, n.bo, sizeof O.bo);
  O.n2_max = n.n2_max;
  return O;
}

template <int H, int FK, int NH, bool F16P>
int launch_one(const LaunchCommon& L, cudaStream_t s) {
  // chains: TMEM 3 x 160 columns at H = 64, 5 x 80 below
  constexpr int NCH = H == 64 ? 3 : 5, NF = 2;
  using S = F32Smem<H, FK, NH, NCH, NF>;
  static_assert(S::BYTES <= 227 * 1024, "shared memory");
  auto k = eval_f32_tc_kernel<H, FK, NH, F16P, NCH, NF>;
  static std::atomic<uint64_t> configured{0};
  once_per_device(configured, [&] {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, S::BYTES);
    const int pct = (S::BYTES + 1024) * 100 / (228 * 1024) + 1;
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
  });
  const int64_t ntiles = (L.n + 127) / 128;
  if (ntiles == 0) return 0;
  const int grid = (int)(ntiles < L.num_sms ? ntiles : L.num_sms);
  k<<<grid, (NCH + NF) * 128, S::BYTES, s>>>(L, f32_params<H>(*L.nw));
  return (int)cudaGetLastError();
}

template <int H, int NH>
int pick(const LaunchCommon& L, cudaStream_t s) {
  const bool f16 = L.pyr.f16 != 0;
  switch (L.shape.frame) {
    case 0: return f16 ? launch_one<H, 0, NH, true>(L, s) : launch_one<H, 0, NH, false>(L, s);
    case 1: return f16 ? launch_one<H, 1, NH, true>(L, s) : launch_one<H, 1, NH, false>(L, s);
    case 2: return f16 ? launch_one<H, 2, NH, true>(L, s) : launch_one<H, 2, NH, false>(L, s);
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace

size_t f32_tc_blob_bytes(const Shape& s) {
  return f16_supported(s) ? (size_t)f32_lay(s.H, s.frame, s.NH).BYTES : 0;
}

int pack_f32_tc_blob(const Shape& s, const float* frame, const float* dec, uint8_t* out, NarrowW* nw) {
  if (!f16_supported(s)) return -1;
  std::memset(nw, 0, sizeof *nw);
  if (s.frame == 1) {
    for (int j = 0; j < 16; ++j) {
      for (int k = 0; k < 8; ++k) nw->f1[k][j] = frame[j * 8 + k];
      nw->fb1[j] = frame[128 + j];
    }
    for (int j = 0; j < 6; ++j) {
      for (int k = 0; k < 16; ++k) nw->f2[j][k] = frame[144 + j * 16 + k];
      nw->fb2[j] = frame[240 + j];
    }
  } else if (s.frame == 2) {
    for (int j = 0; j < 12; ++j) {
      for (int k = 0; k < 8; ++k) nw->f1[k][j] = frame[j * 8 + k];
      nw->fb1[j] = frame[96 + j];
    }
  }
  const int H = s.H;
  const F32Lay o = f32_lay(H, s.frame, s.NH);
  std::memset(out, 0, (size_t)o.BYTES);
  bool ok = true;
  auto put = [&](uint8_t* base, int row, int k, uint16_t v) {
    std::memcpy(base + (k / 8) * (H * 16) + row * 16 + (k % 8) * 2, &v, 2);
  };
  auto put3 = [&](uint8_t* base, int K, int row, int k, float w) {
    uint16_t t[3];
    ok = bf16_split(w, t) && ok;
    for (int b = 0; b < 3 && ok; ++b) put(base + b * H * K * 2, row, k, t[b]);
  };
  const float* p = dec;
  for (int n = 0; n < H; ++n) {
    for (int k = 0; k < s.in; ++k) put3(out + o.B1, o.KX, n, k, p[n * s.in + k]);
    put3(out + o.B1, o.KX, n, s.in, p[H * s.in + n]);
  }
  p += H * s.in + H;
  for (int l = 0; l < s.NH - 1; ++l) {
    uint8_t* b = out + o.BH + l * (3 * H * H + 16 * H) * 2;
    for (int n = 0; n < H; ++n) {
      for (int k = 0; k < H; ++k) put3(b, H, n, k, p[n * H + k]);
      uint16_t t[3];
      ok = bf16_split(p[H * H + n], t) && ok;
      for (int k = 0; k < 3; ++k) put(b + 3 * H * H * 2, n, k, t[k]);
    }
    p += H * H + H;
  }
  for (int n = 0; n < s.out; ++n) {
    for (int k = 0; k < H; ++k) nw->wo[n][k] = p[n * H + k];
    nw->bo[n] = p[s.out * H + n];
  }
  const int widths[5] = {s.in, H, H, s.NH == 3 ? H : s.out, s.out};
  const double n2 = input_limit(dec, widths, s.NH + 1);
  // (inputs within binary16's range: at most 20 of them below 2^16)
  if (!(n2 >= 0x1p37)) ok = false;
  nw->n2_max = n2 < 3e38 ? (float)n2 : 3e38f;
  return ok ? 0 : -1;
}

int launch_eval_f32_tc(const LaunchCommon& L, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  if (!f16_supported(L.shape)) return (int)cudaErrorInvalidValue;
  if (L.shape.NH == 3) return pick<64, 3>(L, s);
  if (L.shape.H == 16) return pick<16, 2>(L, s);
  if (L.shape.H == 32) return pick<32, 2>(L, s);
  return pick<64, 2>(L, s);
}

}  // namespace nam
