// Reverse mode of the FP32 evaluation, the log-space L1 loss and Adam
// (training of the decoder and the latent texture, Sec. 5).
//
// Backward kernel: two groups of eight compute warps each take tiles of 64
// queries, one group's waits under the other's work; the MMAs are issued by
// threads of the compute warps (issuing warps of their own would cost every
// thread 32 of its 128 registers: 453 us against 411).  The forward is recomputed in FP32 on the FMA
// pipes, in a fixed order of operations (a ReLU sign that a rounding flips
// moves a texel's gradient by far more than the rounding); everything behind
// the signs, which is two thirds of the work, runs on the tensor cores as
// bf16 MMAs on three-way splits (x = x_h + x_m + x_l, eight significant bits
// each; six products, FP32 accumulation, small products first), which have
// FP32's range.  The deltas' terms are cut off, the other operand's (weights,
// H1, X, HF) rounded to nearest: the three products left out are below 1.5
// 2^-23 of a term and of either sign (with both cut off up to 3.9 2^-23 of one
// sign).  Weight gradients against 64 bits, as a multiple of the error of every
// product on the FMA pipes (40,000 queries, by layer): 0.70 .. 1.08.
//  - a quad of four adjacent lanes per query: the latent fetch, the frame MLP
//    (lane p owns frame hidden units p + 4e, the six outputs are summed over
//    the quad), the frame construction and its backward (redundant in the
//    quad, ALU only) and the pyramid scatter (lane p takes bilinear tap p;
//    taps that coincide, as at the coarsest levels, are merged so that each
//    distinct texel of a query takes one update);
//  - a half-warp per four queries for the decoder's forward: lane l owns
//    hidden units l + 16 jj of all four queries, a 4 x (H/16) register block,
//    so that every shared-memory operand feeds four FMAs per query block; the
//    output layer's gradient, three columns wide, is summed in these lanes;
//  - MMAs per tile: d1 = D2 W2 (queries in the rows), dx = D1 W1, and, with
//    the same operands read the other way (queries along K), C2 = D2^T [H1 |
//    X 1], C1 = D1^T [X 1] and CF = [DHF | DR]^T [X 1 | HF], which hold every
//    weight and bias gradient of the other layers; they are read back each
//    tile and summed in registers (the accumulator cuts off instead of rounding:
//    a sum over all tiles in it would drift), one atomic per parameter and
//    CTA at the end.  (An infinite delta may give NaN where a product of FP32
//    values would give an infinity.)
// Operand arrays: [term][unit / 8][query][unit % 8] bf16, which is K-major for
// the products over units and MN-major for those over queries.
// What bounds it: the latency of the tile's chain of stages (16 warps a CTA,
// which shared memory and registers allow no more of; the forward on the FMA
// pipes is a fifth of a tile's time, the fetch and the scatter a sixth each).
// H = 64 with the fused loss, 262,144 queries, 1024^2 pyramid: 279 us, against
// 378 us with every product on the FMA pipes; 131,072 queries with the latents
// given: 131 us (163).  Smaller batches and decoders, against that kernel
// (512^2, no loss): H = 64, 10,000 queries 29 us (35); H = 16, 262,144 queries
// 187 us (206), 10,000 queries 20.6 us (22.7), 7,000 without the frame 16.5 us
// (18.6), one query 12.4 us (10.4: the only sizes that lose are single tiles at
// H = 16 and 32 without the frame, to the three MMA round trips).
// Training step variant (LOSS): the decoder blocks also finish the forward
// (y = Wo h2 + bo, summed over the half-warp), evaluate the log-space L1
// loss against the target and start the backward from its gradient, so a
// training step needs no separate forward or loss pass.  With the albedo
// head (ALB: six outputs, RGB then albedo) the fused loss adds the albedo's
// L2 error against one-sample albedo estimates (the paper's albedo
// inference).
// Same-address atomics serialise in L2, and every query whose lod reaches
// the coarsest levels lands on a handful of texels there: the gradient of
// the coarsest levels is summed in shared memory first (per warp for the
// tiniest ones, per CTA for the next) and added to the global buffer once
// per CTA.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace nam {

constexpr int kBwdQ = 64;             // queries per tile, one tile per group
constexpr int kBwdGroup = 4 * kBwdQ;  // threads of a group: a quad per query
constexpr int kBwdThreads = 2 * kBwdGroup;
constexpr int kBlk = kBwdQ * 16;      // bytes of an operand block (eight units of the queries)

template <int H, bool ALB = false>
struct BwdSmem {
  static constexpr int NO = ALB ? 6 : 3;  // decoder outputs
  static constexpr int DW = ALB ? 8 : 4;  // DY row length
  static constexpr int S = H + 4;  // padded row stride of H1
  // operand terms: A holds first D2 (H / 8 blocks), then D1, DHF (2 blocks)
  // and DR (1); B holds H1, X (2 blocks, with the 1) and HF (2).  An MMA's A
  // has 128 rows, a group's 64 (or 24) of them in its half of the TMEM
  // lanes: it reads up to 8 KB before and 16 KB past a term's start, rows
  // whose results are not used, inside this struct.
  static constexpr int TA = (H / 8 + 3) * kBlk, TB = (H / 8 + 4) * kBlk;
  // parameters
  float fW1[16 * 8], fb1[16], fW2[6 * 16], fb2[8];
  // W1 (14 inputs, zero padding) and W2 of the forward's packed FMAs: row 16 p
  // + l holds (w[l + 32 p][k], w[l + 32 p + 16][k]) for every k, or for H = 16
  // w[l][k]; 16 bytes of padding: the rows of a half-warp hit distinct banks
  static constexpr int P = H >= 32 ? 2 : 1;
  static constexpr int S1 = 16 * P + 4, S2 = H * P + 4;
  float W1[H / P][S1];
  float b1[H];
  float W2[H / P][S2];
  float b2[H];
  float Wo[NO * H], bo[8];
  float lred[16];       // per-warp loss partials
  float gwo[NO * H + 8];  // output layer's gradient of the CTA
  uint32_t tslot, pad[3];
  uint64_t bars[8];  // per group: d1, C2, dx, C1
  // per group, of the current tile (deltas at pre-activations)
  struct Group {
    uint32_t mask1[8][16];  // per warp and (jj * 4 + qq): layer-1 signs of its two half-warps
    float R[kBwdQ][8];      // frame MLP output r = (n_raw, t_raw)
    float X[kBwdQ][16];     // decoder input x (14), zero padding; then dL/dx
    float DY[kBwdQ][DW];    // delta at the outputs (after the cosine factor), zero padding;
                            // with the fused loss first the targets and the cosine
                            // factor: (t_r, t_g, t_b, cf), or with ALB (t_r, t_g, t_b,
                            // albedo t_r, t_g, t_b, 0, cf)
    alignas(128) uint8_t A[3 * TA];  // before D2: layer-1 activations H1[q][S] in FP32
    uint8_t B[3 * TB];
  } g[2];
  uint8_t W2T[3 * H * H * 2];   // MMA B operand of d1: rows k, K = j
  uint8_t W1T[3 * 16 * H * 2];  // MMA B operand of dx: rows c, K = j
};

// the three bf16 terms of x (its next eight significant bits each), as bits
__device__ __forceinline__ void split3_one(float x, uint16_t& h, uint16_t& m, uint16_t& l) {
  const uint32_t b = __float_as_uint(x);
  const float r = x - __uint_as_float(b & 0xFFFF0000u);
  const uint32_t br = __float_as_uint(r);
  const float q = r - __uint_as_float(br & 0xFFFF0000u);
  h = (uint16_t)(b >> 16);
  m = (uint16_t)(br >> 16);
  l = (uint16_t)(__float_as_uint(q) >> 16);
}
// the same of x (1 + up), rounded to nearest: terms of either sign, so that what
// the six products leave out (middle times last, last times last) has no sign
// of its own.  `up` makes up for the accumulator, which cuts off
__device__ __forceinline__ void split3_up(float x, float up, uint16_t& h, uint16_t& m, uint16_t& l) {
  const __nv_bfloat16 a = __float2bfloat16_rn(x);
  const float r = x - __bfloat162float(a);
  const __nv_bfloat16 b = __float2bfloat16_rn(r);
  h = __bfloat16_as_ushort(a);
  m = __bfloat16_as_ushort(b);
  l = __bfloat16_as_ushort(__float2bfloat16_rn(fmaf(x, up, r - __bfloat162float(b))));
}
// (measured against 64 bits: dL/dz came out 1.6e-7 too small with cut-off weight
// terms; the weight gradients 1.0e-7 with cut-off terms of both operands,
// 0.6e-7 with those of H1, X and HF rounded, below 0.2e-7 with these factors)
constexpr float kWeightUp = 4e-8f;  // W1, W2 in the products over units
constexpr float kSumUp = 6e-8f;     // H1, X, HF in the products over queries
// U values (consecutive units) of one query to their rows of the three terms;
// p: the first unit's place in term 0, TS: bytes of a term.  RN: terms
// rounded to nearest (split3_rn)
template <int U, int TS, bool RN = false>
__device__ __forceinline__ void put_terms(uint8_t* p, const float (&v)[U]) {
  uint32_t w[3][U / 2];
#pragma unroll
  for (int j = 0; j < U / 2; ++j) {
    if (RN) ptx::split3_rn(v[2 * j], v[2 * j + 1], kSumUp, w[0][j], w[1][j], w[2][j]);
    else ptx::split3(v[2 * j], v[2 * j + 1], w[0][j], w[1][j], w[2][j]);
  }
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    if constexpr (U == 4) {
      *reinterpret_cast<uint2*>(p + t * TS) = make_uint2(w[t][0], w[t][1]);
    } else {
#pragma unroll
      for (int b = 0; b < U / 8; ++b)
        *reinterpret_cast<uint4*>(p + t * TS + b * kBlk) =
            make_uint4(w[t][4 * b], w[t][4 * b + 1], w[t][4 * b + 2], w[t][4 * b + 3]);
    }
  }
}

// Log-space L1 loss of one output element g against its target y (Sec. 5.2
// names an L1 loss in log space; read as |log(1 + max(g, 0)) - log(1 + y)|
// plus 0.01 max(-g, 0), which keeps a gradient on negative outputs); returns
// the loss, *grad = dloss/dg.
__device__ __forceinline__ float log_l1(float g, float y, float* grad) {
  const float d = log1pf(fmaxf(g, 0.0f)) - log1pf(y);
  float l = fabsf(d);
  float gr = 0.0f;
  if (g > 0.0f) gr = (d > 0.0f ? 1.0f : (d < 0.0f ? -1.0f : 0.0f)) / (1.0f + g);
  if (g < 0.0f) {
    l += 0.01f * (-g);
    gr -= 0.01f;
  }
  *grad = gr;
  return l;
}

__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

__device__ __forceinline__ float dot4(const float4 a, const float4 b, float s) {
  s = fmaf(a.x, b.x, s);
  s = fmaf(a.y, b.y, s);
  s = fmaf(a.z, b.z, s);
  return fmaf(a.w, b.w, s);
}

// The latent of a quad's query: lane p filters channels 2p and 2p + 1 (a texel
// is one 32-byte sector of the four lanes' loads).  quad_taps starts the
// loads, quad_filter sums in fetch_latent's order of operations.  f0: u, v,
// lod, xi in lanes 0..3.
struct QuadTaps {
  float2 x[8];
  float w[8];
};
__device__ __forceinline__ void quad_taps(const BackwardArgs& A, float f0, int p, QuadTaps& T) {
  const float u = __shfl_sync(0xffffffffu, f0, 0, 4), v = __shfl_sync(0xffffffffu, f0, 1, 4);
  const float lod = __shfl_sync(0xffffffffu, f0, 2, 4), xi = __shfl_sync(0xffffffffu, f0, 3, 4);
  const LevelPick lp = pick_levels(A.pyr, lod);
  const bool stoch = A.pyr.filter == NAM_FILTER_STOCHASTIC;
  auto level = [&](int l, float wgt, bool load, float2* x, float* w) {
    const int W = A.pyr.w[l];
    int x0, x1, y0, y1;
    float fx, fy;
    tap_axis(A.pyr, u, W, x0, x1, fx);
    tap_axis(A.pyr, v, A.pyr.h[l], y0, y1, fy);
    const uint32_t base = (uint32_t)A.pyr.off[l];
    const uint32_t r0 = base + (uint32_t)y0 * (uint32_t)W, r1 = base + (uint32_t)y1 * (uint32_t)W;
    const uint32_t idx[4] = {r0 + x0, r0 + x1, r1 + x0, r1 + x1};
    const float gx = 1.0f - fx, gy = 1.0f - fy;
    w[0] = gx * gy * wgt;
    w[1] = fx * gy * wgt;
    w[2] = gx * fy * wgt;
    w[3] = fx * fy * wgt;
    const float2* t = reinterpret_cast<const float2*>(A.pyramid) + p;
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = load ? __ldg(t + 4 * (size_t)idx[k]) : make_float2(0.0f, 0.0f);
  };
  level(stoch && xi < lp.t ? lp.l1 : lp.l0, stoch ? 1.0f : 1.0f - lp.t, true, T.x, T.w);
  // (a level of weight 0 is not read and adds zeros)
  level(lp.l1, stoch ? 0.0f : lp.t, !stoch && lp.t != 0.0f, T.x + 4, T.w + 4);
}
__device__ __forceinline__ void quad_gather(float2 a, float z[8]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    z[2 * k] = __shfl_sync(0xffffffffu, a.x, k, 4);
    z[2 * k + 1] = __shfl_sync(0xffffffffu, a.y, k, 4);
  }
}
__device__ __forceinline__ void quad_filter(const QuadTaps& T, float z[8]) {
  float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    acc.x = fmaf(T.w[k], T.x[k].x, acc.x);
    acc.y = fmaf(T.w[k], T.x[k].y, acc.y);
  }
  quad_gather(acc, z);
}

// a[qq][jj] += w[unit jj][4 m ..] . x[qq], in the order of dot4.  P = 2: units
// jj and jj + 1 side by side in packed FMAs (half the FMA instructions, and
// moves that double x; the kernel 290 -> 281 us).  w: this lane's first row, the
// next units' 16 rows of W floats on.
template <int JB, int P, int W>
__device__ __forceinline__ void fma_block(float (&a)[4][JB], const float* w, const float4 (&x)[4], int m) {
  if constexpr (P == 2) {
#pragma unroll
    for (int jj = 0; jj < JB; jj += 2) {
      const float4 w0 = reinterpret_cast<const float4*>(w + 8 * jj * W)[2 * m];
      const float4 w1 = reinterpret_cast<const float4*>(w + 8 * jj * W)[2 * m + 1];
#pragma unroll
      for (int qq = 0; qq < 4; ++qq) {
        float2 s = make_float2(a[qq][jj], a[qq][jj + 1]);
        s = ptx::fma2(make_float2(w0.x, w0.y), make_float2(x[qq].x, x[qq].x), s);
        s = ptx::fma2(make_float2(w0.z, w0.w), make_float2(x[qq].y, x[qq].y), s);
        s = ptx::fma2(make_float2(w1.x, w1.y), make_float2(x[qq].z, x[qq].z), s);
        s = ptx::fma2(make_float2(w1.z, w1.w), make_float2(x[qq].w, x[qq].w), s);
        a[qq][jj] = s.x;
        a[qq][jj + 1] = s.y;
      }
    }
  } else {
#pragma unroll
    for (int jj = 0; jj < JB; ++jj) {
      const float4 v = reinterpret_cast<const float4*>(w + 16 * jj * W)[m];
#pragma unroll
      for (int qq = 0; qq < 4; ++qq) a[qq][jj] = dot4(v, x[qq], a[qq][jj]);
    }
  }
}

// One query's fields, spread over its quad: lane p holds (u, v, lod, xi)[p],
// wi[p], wo[p], and target or output gradient [p] and [3 + p] (p < 3).
struct QuadFields {
  float f0, f1, f2, g0, g1;
};
template <bool LOSS, bool ALB>
__device__ __forceinline__ QuadFields quad_fields(const BackwardArgs& A, int64_t i, bool valid, int p) {
  QuadFields f{};
  const float* a = p == 0 ? A.q.u : p == 1 ? A.q.v : p == 2 ? A.q.lod : A.q.xi;
  if (!A.z_in && a) f.f0 = __ldg(a + i);
  if (p < 3) {
    f.f1 = __ldg((p == 0 ? A.q.wix : p == 1 ? A.q.wiy : A.q.wiz) + i);
    f.f2 = __ldg((p == 0 ? A.q.wox : p == 1 ? A.q.woy : A.q.woz) + i);
    if (valid) {
      if (LOSS) {
        f.g0 = __ldg(A.target + 3 * i + p);
        if (ALB) f.g1 = __ldg(A.target_albedo + 3 * i + p);
      } else {
        f.g0 = __ldg(A.grad_rgb + (ALB ? 6 : 3) * i + p);
        if (ALB) f.g1 = __ldg(A.grad_rgb + 6 * i + 3 + p);
      }
    }
  }
  return f;
}

template <int H, bool FRAME, bool LOSS, bool ALB>
__global__ void __launch_bounds__(kBwdThreads, 1) backward_kernel(const BackwardArgs A) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  using Sm = BwdSmem<H, ALB>;
  Sm& S = *reinterpret_cast<Sm*>(smem_raw);
  constexpr int NO = Sm::NO, DW = Sm::DW, TA = Sm::TA, TB = Sm::TB, P = Sm::P;
  constexpr int JB = H / 16;  // hidden units per lane in the decoder blocks
  constexpr int U = H / 4;    // units per lane where a row is shared by four
  constexpr int N2 = H + 16;  // columns of C2
  // TMEM columns of a group
  constexpr int cD1 = 0, cDX = 64, cC2 = 80, cC1 = 160, cCF = 176, cGroup = 208;
  const int t = threadIdx.x;
  const int lane = t & 31, warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  // groups: compute warps 4k and 4k + 1 (TMEM lanes 0..63), 4k + 2 and 4k + 3
  // (lanes 64..127)
  const int grp = (warp >> 1) & 1;
  typename Sm::Group& G = S.g[grp];
  const uint32_t bar0 = ptx::smem_u32(S.bars) + 32 * grp;
  const int bid = 4 * grp;  // named barriers bid + 1 .. bid + 4
  const int64_t ntiles = (A.n + kBwdQ - 1) / kBwdQ;
  const int64_t tile0 = blockIdx.x + (int64_t)grp * gridDim.x, tstep = 2 * (int64_t)gridDim.x;
  // lw: this warp in its group
  const int lw = ((warp >> 2) << 1) | (warp & 1), lt = 32 * lw + lane;
  const int ql = lt >> 2, p = lt & 3;         // quad: query ql, lane p
  // the fields of the next tile are loaded a tile ahead, the first one's before
  // the parameters (its texels as well would cost more in spilled registers than
  // their latency)
  auto row_of = [&](int64_t tile, bool& valid) -> int64_t {
    const int64_t start = tile * kBwdQ;
    valid = ql < A.n - start;
    return start + (valid ? ql : 0);
  };
  QuadFields nxt{};
  if (tile0 < ntiles) {
    bool v;
    const int64_t i = row_of(tile0, v);
    nxt = quad_fields<LOSS, ALB>(A, i, v, p);
  }
  // ---- parameters -> shared ---------------------------------------------------
  // Every load of a thread is in flight before its first value is used (loops
  // over the arrays one after the other, and the weights read twice, were ten
  // memory latencies: 2,200 to 8,000 cycles of a small batch's 30,000 to 50,000).
  {
    const float* W1 = A.params + (FRAME ? 246 : 0);
    const float* W2 = W1 + 14 * H + H;
    constexpr int kTail = H + NO * H + NO;  // b2, Wo, bo
    static_assert(H * H / 8 <= kBwdThreads && kTail + 8 <= kBwdThreads, "one pass");
    const float vf = FRAME && t < 246 ? __ldg(A.params + t) : 0.0f;
    const float v1 = t < H ? __ldg(W1 + 14 * H + t) : 0.0f;
    const float vt = t < kTail ? __ldg(W2 + H * H + t) : 0.0f;
    // eight units j of one input each
    const int j1 = t / 16 * 8, c1 = t % 16, j2 = t / H * 8, k2 = t % H;
    float w1[8], w2[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      w1[e] = j1 < H && c1 < 14 ? __ldg(W1 + (j1 + e) * 14 + c1) : 0.0f;
      w2[e] = j2 < H ? __ldg(W2 + (j2 + e) * H + k2) : 0.0f;
    }
    for (int i = t; i < NO * H + 8; i += kBwdThreads) S.gwo[i] = 0.0f;
    // fW1, fb1, fW2, fb2, and b2, Wo, bo, lie side by side, zeros behind them
    if (FRAME && t < 248) (&S.fW1[0])[t] = vf;
    if (t < H) S.b1[t] = v1;
    if (t < kTail - NO + 8) (&S.b2[0])[t] = vt;
    auto row = [](int j) { return P == 2 ? (j >> 5) * 16 + (j & 15) : j; };
    auto col = [](int j, int k) { return P == 2 ? 2 * k + ((j >> 4) & 1) : k; };
    // the eight units of a K block side by side in the B operands of the delta
    // products: rows k (or c), K index j
    auto operand = [](uint8_t* o, int term, const float (&w)[8]) {
      uint32_t v[3][4];
#pragma unroll
      for (int e = 0; e < 4; ++e) ptx::split3_rn(w[2 * e], w[2 * e + 1], kWeightUp, v[0][e], v[1][e], v[2][e]);
#pragma unroll
      for (int e = 0; e < 3; ++e) *reinterpret_cast<uint4*>(o + e * term) = make_uint4(v[e][0], v[e][1], v[e][2], v[e][3]);
    };
    if (j1 < H) {
#pragma unroll
      for (int e = 0; e < 8; ++e) S.W1[row(j1 + e)][col(j1 + e, c1)] = w1[e];
      operand(S.W1T + j1 / 8 * 256 + c1 * 16, 16 * H * 2, w1);
    }
    if (j2 < H) {
#pragma unroll
      for (int e = 0; e < 8; ++e) S.W2[row(j2 + e)][col(j2 + e, k2)] = w2[e];
      operand(S.W2T + j2 / 8 * (H * 16) + k2 * 16, H * H * 2, w2);
    }
  }
  if (t == 0) {
    // C1 and CF are issued by two warps
    for (int k = 0; k < 8; ++k) ptx::mbar_init(ptx::smem_u32(&S.bars[k]), (k & 3) == 3 ? 2 : 1);
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_u32(&S.tslot), 512);
    ptx::tmem_relinquish();
  }
  // coarse-level accumulators after the tile: [16 warps][tiny_n][8], [cta_n][8]
  float* wacc = reinterpret_cast<float*>(smem_raw + sizeof(Sm));
  float* cacc = wacc + 16 * 8 * A.tiny_n;
  for (int i = t; i < 8 * (16 * A.tiny_n + A.cta_n); i += kBwdThreads) wacc[i] = 0.0f;
  float* my_wacc = wacc + (t >> 5) * 8 * A.tiny_n;

  ptx::fence_proxy_async();
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = S.tslot + cGroup * grp;
  bool bad = false;

  // A stage's products, one thread: six of term pairs, the small ones first.
  // a, b: the descriptors of the first term's first step
  auto products = [&](uint32_t d, uint64_t a, uint32_t ta, uint32_t astep, uint64_t b, uint32_t tb, uint32_t bstep,
                      int steps, uint32_t id) {
    const int at[6] = {2, 1, 0, 1, 0, 0}, bt[6] = {0, 1, 2, 0, 1, 0};
#pragma unroll
    for (int e = 0; e < 6; ++e)
#pragma unroll
      for (int s = 0; s < steps; ++s)
        ptx::mma_f16(d, ptx::sdesc_at(a, at[e] * ta + s * astep, 0), ptx::sdesc_at(b, bt[e] * tb + s * bstep, 0), id,
                     e + s > 0 ? 1u : 0u);
  };
  // operands: the second group's rows are 64..127 of an MMA
  const uint32_t aA = ptx::smem_u32(G.A), aB = ptx::smem_u32(G.B);
  const uint32_t aK = aA - grp * 64 * 16, aM = aA - grp * 8 * kBlk;
  constexpr uint32_t kMN = (1u << 15) | (1u << 16);  // both operands MN-major
  // gradients of this thread's part of C2, C1 and CF: row grow of the group's
  // half of the TMEM lanes, a quarter of the columns
  const int grow = 32 * (lw & 1) + lane, gq = lw >> 1;
  const uint32_t tl = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
  const bool use2 = 32 * (lw & 1) < H, usef = FRAME && (lw & 1) == 0;
  float acc2[N2 / 4], acc1[4], accf[8], gwo[NO][JB], gbo[NO];
#pragma unroll
  for (int i = 0; i < N2 / 4; ++i) acc2[i] = 0.0f;
#pragma unroll
  for (int i = 0; i < 4; ++i) acc1[i] = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) accf[i] = 0.0f;
#pragma unroll
  for (int c = 0; c < NO; ++c) {
    gbo[c] = 0.0f;
#pragma unroll
    for (int jj = 0; jj < JB; ++jj) gwo[c][jj] = 0.0f;
  }
  // the weight gradients of the tile before: add C2, C1 and CF to the registers
  auto collect = [&]() {
    ptx::tc_fence_after();
    if (use2) {
#pragma unroll
      for (int c0 = 0; c0 < N2 / 4; c0 += 4) {
        uint32_t v[4];
        ptx::tmem_ld4(tl + cC2 + gq * (N2 / 4) + c0, v);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 4; ++e) acc2[c0 + e] += __uint_as_float(v[e]);
      }
      uint32_t v[4];
      ptx::tmem_ld4(tl + cC1 + 4 * gq, v);
      ptx::tmem_ld_wait();
#pragma unroll
      for (int e = 0; e < 4; ++e) acc1[e] += __uint_as_float(v[e]);
    }
    if (usef) {
      uint32_t v[8];
      ptx::tmem_ld8(tl + cCF + 8 * gq, v);
      ptx::tmem_ld_wait();
#pragma unroll
      for (int e = 0; e < 8; ++e) accf[e] += __uint_as_float(v[e]);
    }
  };
  uint32_t ph = 0;  // parity of this tile's MMAs

  float lsum = 0.0f;  // fused loss: this lane's share of the sum
  const int hl = lt & 15, qb = (lt >> 4) * 4;  // half-warp: queries qb..qb+3, units hl + 16 jj
  const bool cosine = (A.flags & NAM_OUT_COSINE) != 0;
  uint32_t issued = 0;  // tiles whose MMAs were issued (the same in the whole group)
  bool stop = false;    // a wait ran out
  for (int64_t tile = tile0; tile < ntiles; tile += tstep, ph ^= 1u) {
    const int64_t start = tile * kBwdQ;
    const int count = (int)((A.n - start) < kBwdQ ? (A.n - start) : kBwdQ);
    bool valid;
    const int64_t i = row_of(tile, valid);
    const QuadFields cur = nxt;
    if (tile + tstep < ntiles) {
      bool v;
      const int64_t j = row_of(tile + tstep, v);
      nxt = quad_fields<LOSS, ALB>(A, j, v, p);
    }
    // ---- quad: latent, frame MLP, frame, decoder input ----------------------
    float hf[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // frame hidden units p + 4e
    {
      float z[8];
      if (A.z_in) {
        // encoder phase (Sec. 5.1): the latent is given, the texture bypassed
        quad_gather(reinterpret_cast<const float2*>(A.z_in + 8 * i)[p], z);
      } else {
        QuadTaps T;
        quad_taps(A, cur.f0, p, T);
        quad_filter(T, z);
      }
      float wi[3], wo[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        wi[c] = __shfl_sync(0xffffffffu, cur.f1, c, 4);
        wo[c] = __shfl_sync(0xffffffffu, cur.f2, c, 4);
      }
      float x[14];
#pragma unroll
      for (int c = 0; c < 8; ++c) x[c] = z[c];
      if (FRAME) {
        // lane p owns frame hidden units p + 4e (rows 8 floats apart in four
        // distinct bank groups)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float4* row = reinterpret_cast<const float4*>(&S.fW1[(p + 4 * e) * 8]);
          const float4 a = row[0], b = row[1];
          float s = S.fb1[p + 4 * e];
          s = dot4(a, make_float4(z[0], z[1], z[2], z[3]), s);
          s = dot4(b, make_float4(z[4], z[5], z[6], z[7]), s);
          hf[e] = fmaxf(s, 0.0f);
        }
        float r[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          float t = 0.0f;
#pragma unroll
          for (int e = 0; e < 4; ++e) t = fmaf(S.fW2[j * 16 + p + 4 * e], hf[e], t);
          r[j] = quad_sum(t) + S.fb2[j];
        }
        const Frame F = build_frame(r);
        to_local(F, wi[0], wi[1], wi[2], x + 8);
        to_local(F, wo[0], wo[1], wo[2], x + 11);
        if (p == 0) {
          reinterpret_cast<float4*>(&G.R[ql][0])[0] = make_float4(r[0], r[1], r[2], r[3]);
          reinterpret_cast<float4*>(&G.R[ql][0])[1] = make_float4(r[4], r[5], 0.0f, 0.0f);
        }
      } else {
        x[8] = wi[0]; x[9] = wi[1]; x[10] = wi[2];
        x[11] = wo[0]; x[12] = wo[1]; x[13] = wo[2];
      }
      if (p == 0) {
        float4* X4 = reinterpret_cast<float4*>(&G.X[ql][0]);
        X4[0] = make_float4(x[0], x[1], x[2], x[3]);
        X4[1] = make_float4(x[4], x[5], x[6], x[7]);
        X4[2] = make_float4(x[8], x[9], x[10], x[11]);
        X4[3] = make_float4(x[12], x[13], 0.0f, 0.0f);
      }
      // DY: the targets and the cosine factor, or the caller's dL/d(output)
      // times that factor (which scales the RGB only)
      const float cf = cosine ? fmaxf(wi[2], 0.0f) : 1.0f;
      if (p < 3) {
        G.DY[ql][p] = LOSS ? cur.g0 : cur.g0 * cf;
        if (ALB) G.DY[ql][3 + p] = cur.g1;
      } else {
        G.DY[ql][DW - 1] = LOSS ? cf : 0.0f;
        if (ALB) G.DY[ql][6] = 0.0f;
      }
    }
    // the MMAs of the tile before have read A and B: their sums to registers
    if (tile != tile0) {
      bad |= !ptx::mbar_wait(bar0 + 24, ph ^ 1u, A.timeout_ns);
      collect();
    }
    __syncwarp();
    // X (with the 1 that meets the bias deltas) and HF as MMA operands
    if (p < 2) {
      const float4 a = reinterpret_cast<const float4*>(&G.X[ql][0])[2 * p];
      const float4 b = reinterpret_cast<const float4*>(&G.X[ql][0])[2 * p + 1];
      const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, p ? 1.0f : b.z, b.w};
      put_terms<8, TB, true>(G.B + (H / 8 + p) * kBlk + ql * 16, v);
    }
    if (FRAME) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        uint16_t w[3];
        split3_up(hf[e], kSumUp, w[0], w[1], w[2]);
        uint8_t* o = G.B + (H / 8 + 2 + (e >> 1)) * kBlk + ql * 16 + ((p + 4 * e) & 7) * 2;
#pragma unroll
        for (int k = 0; k < 3; ++k) *reinterpret_cast<uint16_t*>(o + k * TB) = w[k];
      }
    }
    // ---- half-warp blocks: decoder forward and backward ---------------------
    float (*H1)[Sm::S] = reinterpret_cast<float (*)[Sm::S]>(G.A);
    uint32_t sgn2 = 0;  // lane jj * 4 + qq: layer-2 signs of unit hl + 16 jj, query qq of either half-warp
    {
      float a[4][JB];
      // layer 1 (the forward value of y is not needed: dL/dy comes in)
#pragma unroll
      for (int jj = 0; jj < JB; ++jj)
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) a[qq][jj] = S.b1[hl + 16 * jj];
#pragma unroll
      for (int c4 = 0; c4 < 4; ++c4) {
        float4 xv[4];
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) xv[qq] = reinterpret_cast<const float4*>(&G.X[qb + qq][0])[c4];
        fma_block<JB, P, Sm::S1>(a, &S.W1[hl][0], xv, c4);
      }
#pragma unroll
      for (int jj = 0; jj < JB; ++jj)
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) {
          H1[qb + qq][hl + 16 * jj] = fmaxf(a[qq][jj], 0.0f);
          const uint32_t act = __ballot_sync(0xffffffffu, a[qq][jj] > 0.0f);
          if (lane == jj * 4 + qq) G.mask1[lw][lane] = act;
        }
      __syncwarp();
      // H1 as MMA operand: a quarter of a row per lane (eight rows side by
      // side in each quarter-warp: no bank conflicts)
      {
        const float* row = &H1[8 * lw + (lane & 7)][U * (lane >> 3)];
        float v[U];
#pragma unroll
        for (int k = 0; k < U; k += 4) {
          const float4 x = *reinterpret_cast<const float4*>(row + k);
          v[k] = x.x; v[k + 1] = x.y; v[k + 2] = x.z; v[k + 3] = x.w;
        }
        const int u0 = U * (lane >> 3);
        put_terms<U, TB, true>(G.B + (u0 / 8) * kBlk + (8 * lw + (lane & 7)) * 16 + (u0 % 8) * 2, v);
      }
      // layer 2
#pragma unroll
      for (int jj = 0; jj < JB; ++jj)
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) a[qq][jj] = S.b2[hl + 16 * jj];
#pragma unroll 2
      for (int m = 0; m < H / 4; ++m) {
        float4 hv[4];
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) hv[qq] = reinterpret_cast<const float4*>(&H1[qb + qq][0])[m];
        fma_block<JB, P, Sm::S2>(a, &S.W2[hl][0], hv, m);
      }
      if (LOSS) {
        // output y = Wo relu(a) + bo of the four queries, summed over the
        // half-warp; a lane then takes element mc of query qb + mq: loss and dL/dy (times the cosine factor) into DY
        if constexpr (ALB) {
          float y[4][NO];
#pragma unroll
          for (int qq = 0; qq < 4; ++qq)
#pragma unroll
            for (int c = 0; c < NO; ++c) y[qq][c] = 0.0f;
#pragma unroll
          for (int jj = 0; jj < JB; ++jj) {
            const int j = hl + 16 * jj;
            float o[NO];
#pragma unroll
            for (int c = 0; c < NO; ++c) o[c] = S.Wo[c * H + j];
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
              const float h = fmaxf(a[qq][jj], 0.0f);
#pragma unroll
              for (int c = 0; c < NO; ++c) y[qq][c] = fmaf(o[c], h, y[qq][c]);
            }
          }
#pragma unroll
          for (int off = 1; off < 16; off <<= 1)
#pragma unroll
            for (int qq = 0; qq < 4; ++qq)
#pragma unroll
              for (int c = 0; c < NO; ++c) y[qq][c] += __shfl_xor_sync(0xffffffffu, y[qq][c], off);
          // lane (mq, mc) takes output elements mc and, with ALB, mc + 4 of query qb + mq
          const int mq = hl >> 2, mc = hl & 3;
          float ym[2] = {0.0f, 0.0f};
#pragma unroll
          for (int qq = 0; qq < 4; ++qq)
#pragma unroll
            for (int c = 0; c < NO; ++c) {
              if (qq == mq && c == mc) ym[0] = y[qq][c];
              if (qq == mq && c == mc + 4) ym[1] = y[qq][c];
            }
          float tv[DW];  // targets; the cosine factor last
#pragma unroll
          for (int c4 = 0; c4 < DW / 4; ++c4) {
            const float4 v = reinterpret_cast<const float4*>(&G.DY[qb + mq][0])[c4];
            tv[4 * c4] = v.x; tv[4 * c4 + 1] = v.y; tv[4 * c4 + 2] = v.z; tv[4 * c4 + 3] = v.w;
          }
          const float cf = tv[DW - 1];
          const bool vq = qb + mq < count;
          __syncwarp();
#pragma unroll
          for (int h2 = 0; h2 < DW / 4; ++h2) {
            const int e = mc + 4 * h2;  // output element of this lane
            float tgt = 0.0f;
#pragma unroll
            for (int c = 0; c < NO; ++c)
              if (c == e) tgt = tv[c];
            float d = 0.0f;
            if (e < 3) {
              // BRDF: log-space L1 of the cosine-weighted output
              const float g = (ym[h2] + S.bo[e]) * cf;
              float gr;
              const float l = log_l1(g, tgt, &gr);
              if (vq) lsum += l;
              d = gr * A.loss_inv * cf;
            } else if (e < NO) {
              // albedo head: L2 against the one-sample albedo estimate
              const float r = ym[h2] + S.bo[e] - tgt;
              if (vq) lsum += r * r;
              d = 2.0f * r * A.loss_inv;
            }
            G.DY[qb + mq][e] = vq ? d : 0.0f;
          }
          __syncwarp();
        } else {
          float y[4][3];
#pragma unroll
          for (int qq = 0; qq < 4; ++qq)
#pragma unroll
            for (int c = 0; c < 3; ++c) y[qq][c] = 0.0f;
#pragma unroll
          for (int jj = 0; jj < JB; ++jj) {
            const int j = hl + 16 * jj;
            const float o[3] = {S.Wo[j], S.Wo[H + j], S.Wo[2 * H + j]};
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
              const float h = fmaxf(a[qq][jj], 0.0f);
#pragma unroll
              for (int c = 0; c < 3; ++c) y[qq][c] = fmaf(o[c], h, y[qq][c]);
            }
          }
          // pairs, fours and so on, a lane keeping the queries of its own low
          // bits: lane hl ends with the sums of query hl & 3
          float y2[2][3], ys[3];
#pragma unroll
          for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              const bool o = hl & 1;
              y2[k][c] = (o ? y[2 * k + 1][c] : y[2 * k][c]) +
                         __shfl_xor_sync(0xffffffffu, o ? y[2 * k][c] : y[2 * k + 1][c], 1);
            }
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const bool o = hl & 2;
            ys[c] = (o ? y2[1][c] : y2[0][c]) + __shfl_xor_sync(0xffffffffu, o ? y2[0][c] : y2[1][c], 2);
          }
#pragma unroll
          for (int off = 4; off < 16; off <<= 1)
#pragma unroll
            for (int c = 0; c < 3; ++c) ys[c] += __shfl_xor_sync(0xffffffffu, ys[c], off);
          const int mq = hl & 3, mc = hl >> 2;
          const float ym = mc == 0 ? ys[0] : mc == 1 ? ys[1] : ys[2];
          const float4 tv = *reinterpret_cast<const float4*>(&G.DY[qb + mq][0]);
          __syncwarp();
          if (mc < 3) {
            const float g = (ym + S.bo[mc]) * tv.w;
            float gr;
            const float l = log_l1(g, mc == 0 ? tv.x : mc == 1 ? tv.y : tv.z, &gr);
            const bool vq = qb + mq < count;
            if (vq) lsum += l;
            G.DY[qb + mq][mc] = vq ? gr * A.loss_inv * tv.w : 0.0f;
          } else {
            G.DY[qb + mq][3] = 0.0f;
          }
          __syncwarp();
        }
      }
      // output layer's gradient and the layer-2 signs
      {
        float dyv[4][NO];
#pragma unroll
        for (int qq = 0; qq < 4; ++qq)
#pragma unroll
          for (int c = 0; c < NO; ++c) {
            dyv[qq][c] = G.DY[qb + qq][c];
            gbo[c] += dyv[qq][c];
          }
#pragma unroll
        for (int jj = 0; jj < JB; ++jj)
#pragma unroll
          for (int qq = 0; qq < 4; ++qq) {
            const float h = fmaxf(a[qq][jj], 0.0f);
#pragma unroll
            for (int c = 0; c < NO; ++c) gwo[c][jj] = fmaf(dyv[qq][c], h, gwo[c][jj]);
            const uint32_t act = __ballot_sync(0xffffffffu, a[qq][jj] > 0.0f);
            if (lane == jj * 4 + qq) sgn2 = act;
          }
      }
    }
    // every warp has read its H1 rows: A takes D2
    if (ptx::bar_red_or(bid + 4, kBwdGroup, bad)) {
      stop = true;
      break;
    }
    // ---- layer-2 delta d2 = (Wo^T dy) where the unit is active ---------------
    {
      const int row = lane & 7, q = 8 * lw + row, u0 = U * (lane >> 3);
      const uint32_t bits = __shfl_sync(0xffffffffu, sgn2, (u0 / 16) * 4 + (row & 3)) >> (16 * (row >> 2) + u0 % 16);
      float dy[NO], v[U];
#pragma unroll
      for (int c = 0; c < NO; ++c) dy[c] = G.DY[q][c];
#pragma unroll
      for (int k = 0; k < U; k += 4) {
        float o[NO][4];
#pragma unroll
        for (int c = 0; c < NO; ++c) {
          const float4 w = *reinterpret_cast<const float4*>(&S.Wo[c * H + u0 + k]);
          o[c][0] = w.x; o[c][1] = w.y; o[c][2] = w.z; o[c][3] = w.w;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float d = o[NO - 1][e] * dy[NO - 1];
#pragma unroll
          for (int c = NO - 2; c >= 0; --c) d = fmaf(o[c][e], dy[c], d);
          v[k + e] = (bits >> (k + e)) & 1u ? d : 0.0f;
        }
      }
      put_terms<U, TA>(G.A + (u0 / 8) * kBlk + q * 16 + (u0 % 8) * 2, v);
    }
    ptx::fence_proxy_async();
    ptx::tc_fence_before();
    ++issued;
    // D2 written: d1 = D2 W2 (warp 0), C2 = D2^T [H1 | X 1] (warp 7)
    if (lw == 0) {
      ptx::bar_sync(bid + 1, kBwdGroup);
      if (ptx::elect()) {
        ptx::tc_fence_after();
        products(tmem + cD1, ptx::sdesc(aK, kBlk, 128), TA, 2 * kBlk, ptx::sdesc(ptx::smem_u32(S.W2T), H * 16, 128),
                 H * H * 2, 2 * H * 16, H / 16, ptx::idesc_bf16(128, H));
        ptx::mma_commit(bar0);
      }
      __syncwarp();
    } else if (lw == 7) {
      ptx::bar_sync(bid + 1, kBwdGroup);
      if (ptx::elect()) {
        ptx::tc_fence_after();
        products(tmem + cC2, ptx::sdesc(aM, 128, kBlk), TA, 256, ptx::sdesc(aB, 128, kBlk), TB, 256, kBwdQ / 16,
                 ptx::idesc_bf16(128, N2) | kMN);
        ptx::mma_commit(bar0 + 8);
      }
      __syncwarp();
    } else {
      ptx::bar_arrive(bid + 1, kBwdGroup);
    }
    // ---- layer-1 delta d1 = (W2^T d2) where the unit is active ---------------
    {
      bad |= !ptx::mbar_wait(bar0, ph, A.timeout_ns);
      ptx::tc_fence_after();
      const int u0 = U * gq;
      const uint32_t bits = G.mask1[grow >> 3][(u0 / 16) * 4 + (grow & 3)] >> (16 * ((grow >> 2) & 1) + u0 % 16);
      uint32_t d[U];
#pragma unroll
      for (int k = 0; k < U; k += 4) ptx::tmem_ld4(tl + cD1 + u0 + k, *reinterpret_cast<uint32_t(*)[4]>(&d[k]));
      ptx::tmem_ld_wait();
      float v[U];
#pragma unroll
      for (int k = 0; k < U; ++k) v[k] = (bits >> k) & 1u ? __uint_as_float(d[k]) : 0.0f;
      bad |= !ptx::mbar_wait(bar0 + 8, ph, A.timeout_ns);  // C2 has read D2
      put_terms<U, TA>(G.A + (u0 / 8) * kBlk + grow * 16 + (u0 % 8) * 2, v);
    }
    ptx::fence_proxy_async();
    ptx::tc_fence_before();
    // D1 written: dx = D1 W1 (warp 2), C1 = D1^T [X 1] (warp 6)
    if (lw == 2) {
      ptx::bar_sync(bid + 2, kBwdGroup);
      if (ptx::elect()) {
        ptx::tc_fence_after();
        products(tmem + cDX, ptx::sdesc(aK, kBlk, 128), TA, 2 * kBlk, ptx::sdesc(ptx::smem_u32(S.W1T), 256, 128),
                 16 * H * 2, 512, H / 16, ptx::idesc_bf16(128, 16));
        ptx::mma_commit(bar0 + 16);
      }
      __syncwarp();
    } else if (lw == 6) {
      ptx::bar_sync(bid + 2, kBwdGroup);
      if (ptx::elect()) {
        ptx::tc_fence_after();
        products(tmem + cC1, ptx::sdesc(aM, 128, kBlk), TA, 256, ptx::sdesc(aB + (H / 8) * kBlk, 128, kBlk), TB, 256,
                 kBwdQ / 16, ptx::idesc_bf16(128, 16) | kMN);
        ptx::mma_commit(bar0 + 24);
      }
      __syncwarp();
    } else {
      ptx::bar_arrive(bid + 2, kBwdGroup);
    }
    // ---- dL/dx to its rows ----------------------------------------------------
    if (gq == 0) {
      bad |= !ptx::mbar_wait(bar0 + 16, ph, A.timeout_ns);
      ptx::tc_fence_after();
      uint32_t d[16];
      ptx::tmem_ld16(tl + cDX, d);
      ptx::tmem_ld_wait();
#pragma unroll
      for (int c4 = 0; c4 < 4; ++c4)
        *reinterpret_cast<uint4*>(&G.X[grow][4 * c4]) =
            make_uint4(d[4 * c4], d[4 * c4 + 1], d[4 * c4 + 2], d[4 * c4 + 3]);
      ptx::tc_fence_before();
    }
    if (ptx::bar_red_or(bid + 4, kBwdGroup, bad)) {
      // (the other half of C1's and CF's barrier)
      if (lw == 5 && ptx::elect()) ptx::mma_commit(bar0 + 24);
      stop = true;
      break;
    }
    // ---- quad: frame backward, pyramid scatter --------------------------------
    {
      float dx[16];
#pragma unroll
      for (int c4 = 0; c4 < 4; ++c4) {
        const float4 d = reinterpret_cast<const float4*>(&G.X[ql][0])[c4];
        dx[4 * c4] = d.x; dx[4 * c4 + 1] = d.y; dx[4 * c4 + 2] = d.z; dx[4 * c4 + 3] = d.w;
      }
      float dz[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) dz[c] = dx[c];
      if (FRAME) {
        float r[6];
        {
          const float4 r0 = reinterpret_cast<const float4*>(&G.R[ql][0])[0];
          const float4 r1 = reinterpret_cast<const float4*>(&G.R[ql][0])[1];
          r[0] = r0.x; r[1] = r0.y; r[2] = r0.z; r[3] = r0.w; r[4] = r1.x; r[5] = r1.y;
        }
        const Frame F = build_frame(r);
        // the quantities the frame backward needs
        const float nl = sqrtf(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
        const bool ndeg = !(nl >= 1e-20f);
        const float sdot = r[3] * F.n[0] + r[4] * F.n[1] + r[5] * F.n[2];
        const float tp0 = r[3] - sdot * F.n[0], tp1 = r[4] - sdot * F.n[1], tp2 = r[5] - sdot * F.n[2];
        const float tpl = sqrtf(tp0 * tp0 + tp1 * tp1 + tp2 * tp2);
        const float trl = sqrtf(r[3] * r[3] + r[4] * r[4] + r[5] * r[5]);
        const bool tdeg = !(tpl > 1e-6f * trl);
        const float c0_ = F.n[1] * F.t[2] - F.n[2] * F.t[1];
        const float c1_ = F.n[2] * F.t[0] - F.n[0] * F.t[2];
        const float c2_ = F.n[0] * F.t[1] - F.n[1] * F.t[0];
        const float cl = sqrtf(c0_ * c0_ + c1_ * c1_ + c2_ * c2_);
        float wi[3], wo[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          wi[c] = __shfl_sync(0xffffffffu, cur.f1, c, 4);
          wo[c] = __shfl_sync(0xffffffffu, cur.f2, c, 4);
        }
        // x' = T w: dT row k += dx'_k w
        float dt[3], db[3], dn[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          dt[k] = dx[8] * wi[k] + dx[11] * wo[k];
          db[k] = dx[9] * wi[k] + dx[12] * wo[k];
          dn[k] = dx[10] * wi[k] + dx[13] * wo[k];
        }
        // b = c / |c|, c = n x t
        const float bdb = F.b[0] * db[0] + F.b[1] * db[1] + F.b[2] * db[2];
        const float icl = 1.0f / cl;
        float gc[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) gc[k] = (db[k] - F.b[k] * bdb) * icl;
        dn[0] += F.t[1] * gc[2] - F.t[2] * gc[1];
        dn[1] += F.t[2] * gc[0] - F.t[0] * gc[2];
        dn[2] += F.t[0] * gc[1] - F.t[1] * gc[0];
        dt[0] += gc[1] * F.n[2] - gc[2] * F.n[1];
        dt[1] += gc[2] * F.n[0] - gc[0] * F.n[2];
        dt[2] += gc[0] * F.n[1] - gc[1] * F.n[0];
        float dr[6] = {0, 0, 0, 0, 0, 0};
        if (!tdeg) {
          const float tdt = F.t[0] * dt[0] + F.t[1] * dt[1] + F.t[2] * dt[2];
          const float itpl = 1.0f / tpl;
          float dtp[3];
#pragma unroll
          for (int k = 0; k < 3; ++k) dtp[k] = (dt[k] - F.t[k] * tdt) * itpl;
          const float ndtp = F.n[0] * dtp[0] + F.n[1] * dtp[1] + F.n[2] * dtp[2];
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            dr[3 + k] += dtp[k] - F.n[k] * ndtp;
            dn[k] += -ndtp * r[3 + k] - sdot * dtp[k];
          }
        }
        if (!ndeg) {
          const float ndn = F.n[0] * dn[0] + F.n[1] * dn[1] + F.n[2] * dn[2];
          const float inl = 1.0f / nl;
#pragma unroll
          for (int k = 0; k < 3; ++k) dr[k] += (dn[k] - F.n[k] * ndn) * inl;
        }
        if (!valid) {
#pragma unroll
          for (int k = 0; k < 6; ++k) dr[k] = 0.0f;
        }
        // frame hidden delta, own units p + 4e, and its share of dz
        float dhf[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float g = 0.0f;
#pragma unroll
          for (int j = 0; j < 6; ++j) g = fmaf(S.fW2[j * 16 + p + 4 * e], dr[j], g);
          dhf[e] = hf[e] > 0.0f ? g : 0.0f;
          uint16_t w[3];
          split3_one(dhf[e], w[0], w[1], w[2]);
          uint8_t* o = G.A + (H / 8 + (e >> 1)) * kBlk + ql * 16 + ((p + 4 * e) & 7) * 2;
#pragma unroll
          for (int k = 0; k < 3; ++k) *reinterpret_cast<uint16_t*>(o + k * TA) = w[k];
        }
        if (p == 0) {
          const float v[8] = {dr[0], dr[1], dr[2], dr[3], dr[4], dr[5], 0.0f, 0.0f};
          put_terms<8, TA>(G.A + (H / 8 + 2) * kBlk + ql * 16, v);
        }
        float gz[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) gz[c] = 0.0f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float4* row = reinterpret_cast<const float4*>(&S.fW1[(p + 4 * e) * 8]);
          const float4 a = row[0], b = row[1];
          gz[0] = fmaf(a.x, dhf[e], gz[0]); gz[1] = fmaf(a.y, dhf[e], gz[1]);
          gz[2] = fmaf(a.z, dhf[e], gz[2]); gz[3] = fmaf(a.w, dhf[e], gz[3]);
          gz[4] = fmaf(b.x, dhf[e], gz[4]); gz[5] = fmaf(b.y, dhf[e], gz[5]);
          gz[6] = fmaf(b.z, dhf[e], gz[6]); gz[7] = fmaf(b.w, dhf[e], gz[7]);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) dz[c] += quad_sum(gz[c]);
      }
      // DHF, DR written: CF = [DHF | DR]^T [X 1 | HF] (warp 5), which runs
      // while the texels take their gradients
      ptx::fence_proxy_async();
      ptx::tc_fence_before();
      if (lw == 5) {
        ptx::bar_sync(bid + 3, kBwdGroup);
        if (ptx::elect()) {
          ptx::tc_fence_after();
          if (FRAME)
            products(tmem + cCF, ptx::sdesc(aM + (H / 8) * kBlk, 128, kBlk), TA, 256,
                     ptx::sdesc(aB + (H / 8) * kBlk, 128, kBlk), TB, 256, kBwdQ / 16, ptx::idesc_bf16(128, 32) | kMN);
          ptx::mma_commit(bar0 + 24);
        }
        __syncwarp();
      } else {
        ptx::bar_arrive(bid + 3, kBwdGroup);
      }
      const float u = __shfl_sync(0xffffffffu, cur.f0, 0, 4), v = __shfl_sync(0xffffffffu, cur.f0, 1, 4);
      const float lod = __shfl_sync(0xffffffffu, cur.f0, 2, 4), xi = __shfl_sync(0xffffffffu, cur.f0, 3, 4);
      if (A.dz_out) {
        // encoder phase: dL/dz goes to the encoder's backward
        if (valid && p == 0) {
          reinterpret_cast<float4*>(A.dz_out + 8 * i)[0] = make_float4(dz[0], dz[1], dz[2], dz[3]);
          reinterpret_cast<float4*>(A.dz_out + 8 * i)[1] = make_float4(dz[4], dz[5], dz[6], dz[7]);
        }
      } else if (valid && A.grad_pyramid) {
        // pyramid scatter: z = sum_k w_k texel_k  =>  dtexel_k += w_k dz
        LevelPick lp = pick_levels(A.pyr, lod);
        int lv[2];
        float lw[2];
        int nl2;
        if (A.pyr.filter == NAM_FILTER_STOCHASTIC) {
          lv[0] = xi < lp.t ? lp.l1 : lp.l0;
          lw[0] = 1.0f;
          nl2 = 1;
        } else {
          lv[0] = lp.l0; lw[0] = 1.0f - lp.t;
          lv[1] = lp.l1; lw[1] = lp.t;
          nl2 = lp.t != 0.0f ? 2 : 1;
        }
        for (int e = 0; e < nl2; ++e) {
          const int l = lv[e];
          const int W = A.pyr.w[l], Hh = A.pyr.h[l];
          int x0, x1, y0, y1;
          float fx, fy;
          tap_axis(A.pyr, u, W, x0, x1, fx);
          tap_axis(A.pyr, v, Hh, y0, y1, fy);
          // lane p takes tap p = (y bit, x bit) and the weights of every later
          // tap on the same texel; a tap already taken by an earlier lane is skipped
          int tx[4];
          float tw[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            tx[k] = ((k & 2) ? y1 : y0) * W + ((k & 1) ? x1 : x0);
            tw[k] = ((k & 1) ? fx : 1.0f - fx) * ((k & 2) ? fy : 1.0f - fy);
          }
          const int mine = p == 0 ? tx[0] : p == 1 ? tx[1] : p == 2 ? tx[2] : tx[3];
          bool first = true;
          float w = 0.0f;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (tx[k] == mine) {
              if (k < p) first = false;
              else w += tw[k];
            }
          }
          if (!first) continue;
          w *= lw[e];
          const int64_t tex = A.pyr.off[l] + mine;
          if (tex >= A.cta_tex0) {
            float* c = tex >= A.tiny_tex0 ? my_wacc + 8 * (tex - A.tiny_tex0) : cacc + 8 * (tex - A.cta_tex0);
#pragma unroll
            for (int k = 0; k < 8; ++k) atomicAdd(c + k, w * dz[k]);
          } else {
            float4* g = reinterpret_cast<float4*>(A.grad_pyramid + tex * 8);
            atomicAdd(g, make_float4(w * dz[0], w * dz[1], w * dz[2], w * dz[3]));
            atomicAdd(g + 1, make_float4(w * dz[4], w * dz[5], w * dz[6], w * dz[7]));
          }
        }
      }
    }
  }
  // ---- flush: one atomic per parameter and coarse texel channel per CTA -------
  if (stop) {
    bad = true;
    // the encoder's backward reads every row of dz: those of this group's tiles
    // become zero, so that none is left from an earlier batch (worked out anew
    // here: values kept for this over the loop cost the kernel 10 us in spills)
    if (A.dz_out) {
      const int w = threadIdx.x >> 5, g = (w >> 1) & 1;
      const int r = 32 * (((w >> 2) << 1) | (w & 1)) + (threadIdx.x & 31);
      for (int64_t k = blockIdx.x + (int64_t)g * gridDim.x; k * kBwdQ < A.n; k += 2 * (int64_t)gridDim.x)
        if (k * kBwdQ + (r >> 2) < A.n)
          reinterpret_cast<float2*>(A.dz_out)[4 * k * kBwdQ + r] = make_float2(0.0f, 0.0f);
    }
  } else if (tile0 < ntiles) {
    bad |= !ptx::mbar_wait(bar0 + 24, ph ^ 1u, A.timeout_ns);
    collect();
  }
  if (LOSS) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
    if (lane == 0) S.lred[warp] = lsum;
  }
#pragma unroll
  for (int c = 0; c < NO; ++c) {
#pragma unroll
    for (int jj = 0; jj < JB; ++jj) atomicAdd(&S.gwo[c * H + hl + 16 * jj], gwo[c][jj]);
    if (hl == 0) atomicAdd(&S.gwo[NO * H + c], gbo[c]);
  }
  if (!__syncthreads_or(bad)) {
    if (LOSS && t == 0) {
      float tot = 0.0f;
      for (int w = 0; w < 16; ++w) tot += S.lred[w];
      atomicAdd(A.loss_acc, tot * A.loss_inv);
    }
    // (half a texel at a time: a float at a time, 36,000 of them at H = 16, took
    // 3,700 cycles)
    auto add4 = [](float* g, const float4& c) {
      if (c.x != 0.0f || c.y != 0.0f || c.z != 0.0f || c.w != 0.0f) atomicAdd(reinterpret_cast<float4*>(g), c);
    };
    for (int k = t; k < 2 * A.tiny_n && t < 64; k += 64) {
      float4 c = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      for (int w = 0; w < 16; ++w) {
        const float4 v = reinterpret_cast<const float4*>(wacc + w * 8 * A.tiny_n)[k];
        c = make_float4(c.x + v.x, c.y + v.y, c.z + v.z, c.w + v.w);
      }
      add4(A.grad_pyramid + A.tiny_tex0 * 8 + 4 * k, c);
    }
#pragma unroll 4
    for (int k = t - 64; k < 2 * A.cta_n && t >= 64; k += kBwdThreads - 64)
      add4(A.grad_pyramid + A.cta_tex0 * 8 + 4 * k, reinterpret_cast<const float4*>(cacc)[k]);
    // Both groups' sums of C2, C1 and CF meet in shared memory (odd row
    // lengths: no bank conflicts; the first group's operands are done with),
    // so that the atomics run along the parameters and once per CTA (straight
    // from the registers, a row per lane, they took 20 us more).
    constexpr int R2 = N2 + 1, R1 = 17, RF = 33;
    float* s2 = reinterpret_cast<float*>(S.g[0].A);
    float* s1 = s2 + H * R2;
    float* sf = s1 + H * R1;
    static_assert((H * (R2 + R1) + 22 * RF) * 4 <= 3 * TA, "the sums do not fit");
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (grp == k) {
        auto put = [&](float* d, float v) { *d = k ? *d + v : v; };
        if (grow < H) {
#pragma unroll
          for (int c = 0; c < N2 / 4; ++c) put(s2 + grow * R2 + gq * (N2 / 4) + c, acc2[c]);
#pragma unroll
          for (int c = 0; c < 4; ++c) put(s1 + grow * R1 + gq * 4 + c, acc1[c]);
        }
        if (FRAME && grow < 22) {
#pragma unroll
          for (int c = 0; c < 8; ++c) put(sf + grow * RF + gq * 8 + c, accf[c]);
        }
      }
      __syncthreads();
    }
    float* g = A.grad_params;
    constexpr int o = FRAME ? 246 : 0;
    constexpr int ob1 = o + 14 * H, oW2 = ob1 + H, ob2 = oW2 + H * H, oWo = ob2 + H;
    if (FRAME) {
      // rows: DHF, DR; columns: X (the 1 in column 14), HF
      for (int k = t; k < 246; k += kBwdThreads)
        atomicAdd(&g[k], k < 128   ? sf[(k >> 3) * RF + (k & 7)]
                         : k < 144 ? sf[(k - 128) * RF + 14]
                         : k < 240 ? sf[(16 + (k - 144) / 16) * RF + 16 + (k - 144) % 16]
                                   : sf[(k - 224) * RF + 14]);
    }
    for (int k = t; k < 14 * H; k += kBwdThreads) atomicAdd(&g[o + k], s1[k / 14 * R1 + k % 14]);
    for (int k = t; k < H; k += kBwdThreads) {
      atomicAdd(&g[ob1 + k], s1[k * R1 + 14]);
      atomicAdd(&g[ob2 + k], s2[k * R2 + H + 14]);
    }
    for (int k = t; k < H * H; k += kBwdThreads) atomicAdd(&g[oW2 + k], s2[k / H * R2 + k % H]);
    for (int k = t; k < NO * H + NO; k += kBwdThreads) atomicAdd(&g[oWo + k], S.gwo[k]);  // weights, then the bias
  }

  // ---- teardown ----------------------------------------------------------------
  // MMAs in flight after a wait gave up are waited for with the fixed drain
  // limit, and TMEM is freed only if they completed.
  bool drained = true;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (issued > 0) drained &= ptx::mbar_wait(bar0 + 8 * k, (issued - 1) & 1u, ptx::kDrainTimeoutNs);
  if (bad) {
    record_error(A.err, DEVERR_WAIT_TIMEOUT);
    if (A.failed) atomicExch(A.failed, 1);
  }
  if (!drained) record_error(A.err, DEVERR_DRAIN_TIMEOUT);
  ptx::tc_fence_before();
  const bool all_drained = __syncthreads_and(drained ? 1 : 0) != 0;
  if (warp == 0 && all_drained) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(S.tslot, 512);
  }
}

template <int H, bool FRAME, bool LOSS, bool ALB>
static int launch_bwd_one(const BackwardArgs& a, cudaStream_t s) {
  auto k = backward_kernel<H, FRAME, LOSS, ALB>;
  constexpr int kSmemMax = 227 * 1024;
  constexpr int kBase = (int)sizeof(BwdSmem<H, ALB>);
  static_assert(kBase <= kSmemMax, "backward tile does not fit in shared memory");
  const int64_t tiles = (a.n + kBwdQ - 1) / kBwdQ;
  // a tile per CTA while there are SMs; beyond that a CTA's two groups take one
  // each (its time is theirs, and there are no more sums to add up than needed:
  // with a CTA on every SM 157 tiles took as long and sent twice the atomics,
  // whose roundings made the weight gradients' error 1.3 times as large)
  const int64_t pairs = (tiles + 1) / 2;
  int grid = (int)(tiles <= a.num_sms ? tiles : pairs < a.num_sms ? pairs : a.num_sms);
  if (grid < 1) grid = 1;
  // coarse-level accumulators in what the tile leaves: per-warp copies of the
  // coarsest levels up to kTiny texels, then one copy of the next levels, as long
  // as a CTA's queries (four texels each) can meet there: a copy of 4,000 texels
  // for 64 queries costs more to clear and to look through than their atomics
  constexpr int64_t kTiny = 24;
  BackwardArgs b = a;
  b.tiny_tex0 = b.cta_tex0 = a.pyr.texels;
  b.tiny_n = b.cta_n = 0;
  if (a.grad_pyramid) {
    int64_t room = (kSmemMax - kBase) / 32;  // texels of 8 floats
    int l = a.pyr.levels - 1;
    for (; l >= 0; --l) {
      const int64_t cum = a.pyr.texels - a.pyr.off[l];
      if (cum > kTiny || 16 * cum > room) break;
      b.tiny_tex0 = a.pyr.off[l];
    }
    b.tiny_n = (int32_t)(a.pyr.texels - b.tiny_tex0);
    room -= 16 * (int64_t)b.tiny_n;
    b.cta_tex0 = b.tiny_tex0;
    const int64_t per_cta = a.n / grid;
    for (; l >= 0 && b.tiny_tex0 - a.pyr.off[l] <= room; --l) {
      if ((int64_t)a.pyr.w[l] * a.pyr.h[l] > 2 * per_cta) break;
      b.cta_tex0 = a.pyr.off[l];
    }
    b.cta_n = (int32_t)(b.tiny_tex0 - b.cta_tex0);
  }
  const int smem = kBase + 32 * (16 * b.tiny_n + b.cta_n);
  static std::atomic<uint64_t> attr_done{0};
  once_per_device(attr_done, [&] { cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax); });
  k<<<grid, kBwdThreads, smem, s>>>(b);
  return (int)cudaGetLastError();
}

// Trainable materials keep FP32 latents (the pyramid is an Adam master).
template <int H, bool ALB>
static int bwd_dispatch_alb(const BackwardArgs& a, cudaStream_t s) {
  if (a.target)
    return a.shape.frame ? launch_bwd_one<H, true, true, ALB>(a, s)
                         : launch_bwd_one<H, false, true, ALB>(a, s);
  return a.shape.frame ? launch_bwd_one<H, true, false, ALB>(a, s)
                       : launch_bwd_one<H, false, false, ALB>(a, s);
}

template <int H>
static int bwd_dispatch(const BackwardArgs& a, cudaStream_t s) {
  if (a.pyr.f16) return (int)cudaErrorInvalidValue;
  if (a.shape.out == 6) {
    if (a.target && !a.target_albedo) return (int)cudaErrorInvalidValue;
    return bwd_dispatch_alb<H, true>(a, s);
  }
  return bwd_dispatch_alb<H, false>(a, s);
}

int launch_backward(const BackwardArgs& a, void* stream) {
  if (a.n == 0) return 0;
  cudaStream_t s = (cudaStream_t)stream;
  if (a.shape.NH != 2) return (int)cudaErrorInvalidValue;
  if (a.shape.H == 16) return bwd_dispatch<16>(a, s);
  if (a.shape.H == 32) return bwd_dispatch<32>(a, s);
  if (a.shape.H == 64) return bwd_dispatch<64>(a, s);
  return (int)cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// loss: L = mean |log(1+max(g,0)) - log(1+y)| + 0.01 mean max(-g,0)
// ---------------------------------------------------------------------------
__global__ void loss_kernel(const float* __restrict__ g, const float* __restrict__ y, int64_t m, float inv,
                            float* __restrict__ dg, float* __restrict__ acc) {
  float local = 0.0f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    float grad;
    local += log_l1(g[i], y[i], &grad);
    dg[i] = grad * inv;
  }
  for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
  __shared__ float red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = local;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0f;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) atomicAdd(acc, v * inv);
  }
}

int launch_loss(const float* rgb, const float* target, int64_t n, float* grad_rgb, float* loss_accum, void* stream) {
  const int64_t m = 3 * n;
  if (m == 0) return 0;
  int grid = (int)((m + 255) / 256);
  if (grid > 1024) grid = 1024;
  loss_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(rgb, target, m, 1.0f / (float)m, grad_rgb, loss_accum);
  return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Adam (Kingma & Ba): bias-corrected first and second moments; the gradient
// buffer is cleared after use so the next backward accumulates afresh.
// ---------------------------------------------------------------------------
struct AdamStep {
  float lr, b1, b2, eps, c1, c2;
};

// (a step whose backward failed only clears the gradient, a part of its sum)
__device__ __forceinline__ void adam_one(float& p, float& g, float& m, float& v, const AdamStep& a) {
  const float gi = g;
  m = a.b1 * m + (1.0f - a.b1) * gi;
  v = a.b2 * v + (1.0f - a.b2) * gi * gi;
  p -= a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
  g = 0.0f;
}

__global__ void adam_kernel(float* __restrict__ p, float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                            int64_t count, const AdamStep a, const int* __restrict__ failed) {
  const bool skip = failed && *failed;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    if (skip) g[i] = 0.0f;
    else adam_one(p[i], g[i], m[i], v[i], a);
  }
}

// 16-byte vector form of the same per-element update, bound by HBM: four
// streams read, three written, and the gradient cleared only where a query
// reached the texel (262,144 queries, training step with a 2048^2 pyramid 557
// -> 544 us, 1024^2 384 -> 381, 256^2, where all are reached, the same).
__global__ void adam4_kernel(float4* __restrict__ p, float4* __restrict__ g, float4* __restrict__ m,
                             float4* __restrict__ v, int64_t count4, const AdamStep a,
                             const int* __restrict__ failed) {
  if (failed && *failed) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count4; i += (int64_t)gridDim.x * blockDim.x)
      g[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    return;
  }
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count4; i += (int64_t)gridDim.x * blockDim.x) {
    float4 P = p[i], G = g[i], M = m[i], V = v[i];
    const bool clear = (__float_as_uint(G.x) | __float_as_uint(G.y) | __float_as_uint(G.z) | __float_as_uint(G.w)) != 0;
    adam_one(P.x, G.x, M.x, V.x, a);
    adam_one(P.y, G.y, M.y, V.y, a);
    adam_one(P.z, G.z, M.z, V.z, a);
    adam_one(P.w, G.w, M.w, V.w, a);
    p[i] = P;
    if (clear) g[i] = G;
    m[i] = M;
    v[i] = V;
  }
}

int launch_adam(float* p, const float* g, float* m, float* v, int64_t count, float lr, float b1, float b2, float eps,
                int step, const int* failed, void* stream) {
  if (count == 0) return 0;
  cudaStream_t s = (cudaStream_t)stream;
  const AdamStep a{lr, b1, b2, eps, 1.0f - powf(b1, (float)step), 1.0f - powf(b2, (float)step)};
  float* gm = const_cast<float*>(g);
  int64_t head = 0;
  // small arrays (the MLP masters) in one scalar launch
  if (count >= (1 << 16) && (((uintptr_t)p | (uintptr_t)g | (uintptr_t)m | (uintptr_t)v) & 15u) == 0) {
    const int64_t count4 = count / 4;
    if (count4 > 0) {
      int grid = (int)((count4 + 255) / 256);
      if (grid > 8192) grid = 8192;
      adam4_kernel<<<grid, 256, 0, s>>>(reinterpret_cast<float4*>(p), reinterpret_cast<float4*>(gm),
                                        reinterpret_cast<float4*>(m), reinterpret_cast<float4*>(v), count4, a, failed);
    }
    head = 4 * count4;
  }
  const int64_t rest = count - head;
  if (rest > 0) {
    int grid = (int)((rest + 255) / 256);
    if (grid > 4096) grid = 4096;
    adam_kernel<<<grid, 256, 0, s>>>(p + head, gm + head, m + head, v + head, rest, a, failed);
  }
  return (int)cudaGetLastError();
}

}  // namespace nam
