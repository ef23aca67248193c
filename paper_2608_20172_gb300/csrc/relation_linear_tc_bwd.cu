// relation_linear_tc_bwd.cu -- chunked tensor-core backward of Linear Relation (Sec. 5.2,
// App. A.4; the paper writes out the forward only), bf16, d_h = 64.
//
// Reverse mode through the 128-token blocks of relation_linear_tc.cu, every block in
// parallel.  The state passes come first (relation_linear_tc.cu, launch_states): the blocks'
// contributions to the state and to its adjoint in one launch, then the scans of the state
// C_0 entering every block and of the adjoint dC leaving it,
// dC(b - 1) = Diag(a_L(b)) dC(b) + Qs_b^T dY_b.  Then one CTA per block, with G = dY, A = tril(Qm Km^T, -1), dA = tril(G I~^T, -1):
//   X  = dA Km + G (2^{L_m} C_0)^T        dq'_t = 2^{L_t - L_m} X_t
//   Y  = dA^T Qm + Ys,  Ys = I~ (2^{L_end - L_m} dC)^T   dk'_j = 2^{L_m - L_j} Y_j
//   dI~ = G + A^T G + KL dC
//   dL_t = q'_t * dq'_t - k'_t * dk'_t = Qm_t * X_t - Km_t * Y_t
//          (+ sum_n dC[c][n] C_L[c][n] at the block's end, C_L = 2^{L_end} C_0 + KL^T I~,
//           taken as sum_n (2^{L_m} C_0)[c][n] (2^{L_end - L_m} dC)[c][n] + sum_j Km_j * Ys_j)
//   dalpha_u = (sum_{t >= u} dL_t) / alpha_u           (L_t = sum_{u <= t} log2 alpha_u)
// (the midpoint L_m cancels in every product S_tj, so it carries no gradient), and dp1,
// dp2 from dq', dk' through S_t and the normalisation of p1, p2.
// The suffix sums of dL cancel: every pair (t, j) with both tokens at or after u enters
// once through Qm_t X_t and once, negated, through Km_j Y_j, and every Km_j Ys_j once in the
// end term; only the pairs that straddle u survive, and those carry the factor alpha_u that
// the division takes out.  So dL is formed from the very bf16 values of Qm and Km that the
// products read (recomputed bit for bit), and the end term from the same Ys: the pairs
// then cancel up to fp32 rounding, where rounding Qm and Km independently of q' and k'
// would leave errors of the bf16 unit, divided by alpha_u.  The products are tcgen05
// MMAs with fp32 accumulation in TMEM; the masked A and dA go through shared memory so that
// the transposed products read them as MN-major operands.  Four warpgroups do the
// elementwise work (thread = token; the groups split the channels or columns; the sums whose
// rounding the cancellation above rests on stay one chain each, in the order of the block's
// tokens or channels, on different groups), then a warp the TMA loads and one (warp-uniform,
// elect.sync) the MMAs.  One CTA per SM (220 KB), so latency bounds it: a block's phases and
// barriers around small products, nothing else resident.  B 8, H 12, T 2048, the whole backward:
// 535 us with one elementwise warpgroup and four state launches, 270 with four groups and two,
// 254 with p1 and p2 kept in registers past Qm and Km (they were loaded again) and the small
// retentions' fix-up beside the products, 228 with fewer instructions per element, the state
// pass's blocks shared out among resident CTAs and launches that overlap.  (Persistent CTAs here,
// the next block's tiles loaded early: the same; the registers spill.)
// Every mbarrier wait is bounded (common.cuh); a warp whose wait gave up keeps meeting the
// warpgroups' barriers and skips the work between them.
#include "relation_linear_tc.cuh"

namespace rel {
namespace lintc {
namespace bwd {

constexpr int D = 64;
constexpr int NG = 4;                      // elementwise warpgroups
constexpr int EW = NG * 128, W_TMA = NG * 4, W_MMA = W_TMA + 1, kThreads = EW + 64;
constexpr int kTmemCols = 512;  // scratch S / dA 128 | X 64 | Y 64 | dI~ 64 | Ys 64
constexpr int COL_SC = 0, COL_X = 128, COL_Y = 192, COL_DI = 256, COL_YS = 320;
// shared memory (bytes): 128-token tiles of 64 bf16 columns are 16 KB
constexpr int T16 = LT * 64 * 2;
constexpr int OFF_P1 = 0;                 // p1, then Qm in place, then dp1
constexpr int OFF_P2 = OFF_P1 + T16;      // p2, then Km in place, then dp2
constexpr int OFF_V = OFF_P2 + T16;       // I~
constexpr int OFF_G = OFF_V + T16;        // dY, then dI~ (the dv output)
constexpr int OFF_AL = OFF_G + T16;       // alpha, then its running log2 sums [2][128][32] fp32
constexpr int OFF_KL = OFF_AL + LT * 64 * 4;  // KL; from the epilogue on, dL and Km Ys [t][GS]
constexpr int OFF_AS = OFF_KL + T16;      // A = tril(S) [t][j] (2 blocks), then dL [t][64] fp32
constexpr int OFF_DAS = OFF_AS + 2 * T16; // dA [t][j]
constexpr int C64 = 64 * 64 * 2;          // a [64 c][64 n] bf16 tile
constexpr int OFF_C0 = OFF_DAS + 2 * T16; // C_0, then 2^{L_m} C_0 in place
constexpr int OFF_DC = OFF_C0 + C64;      // dC (the state's adjoint leaving the block)
constexpr int OFF_DCP = OFF_DC + C64;     // 2^{L_end - L_m} dC
constexpr int OFF_SC = OFF_DCP + C64;     // scalars, 15 x 128 fp32
constexpr int kFix = 16;
constexpr int OFF_COEF = OFF_SC + 15 * LT * 4;  // [kFix][128] fp32: Km / Qm of the fix-ups
constexpr int OFF_BAR = OFF_COEF + kFix * LT * 4;
constexpr int SMEM = OFF_BAR + 128 + 1024;
static_assert(SMEM <= 232448, "shared memory");
constexpr uint32_t LOAD_BYTES = 4 * T16 + LT * 64 * 4 + 2 * C64;
constexpr int GS = 68;  // row stride (floats) of the epilogue's [t][64] arrays: float4 rows
constexpr int OFF_GL = OFF_KL, OFF_TS = OFF_GL + LT * GS * 4;
static_assert(OFF_TS + LT * GS * 4 <= OFF_C0, "epilogue arrays overlap the state tiles");

__device__ __forceinline__ float dm_of(float lv, float lm, bool later, bool& clamped) {
  // log2 of a_t / a_m for one channel from its stored running sum (relative to the block's
  // start, or in the later half to the midpoint) and L_m, clamped to +-kClampLog2
  float dm = (lv + (later ? lm : 0.f)) - lm;
  if (fabsf(dm) > kClampLog2) {
    dm = copysignf(kClampLog2, dm);
    clamped = true;
  }
  return dm;
}
// Retention below this takes dalpha from the state and its adjoint at the token (fix_up).
constexpr float kSmallAlpha = 1.0f / 1024.0f;

// A block with more than kFix (token, channel)s of small retention fixes them up at the end,
// from dY, p1 and p2 loaded again over the epilogue's dL and Km Ys arrays once the suffix sums
// are out, and after them the list of the (token, channel)s.
constexpr int OFF_FIX_G = OFF_KL, OFF_FIX_P1 = OFF_KL + T16, OFF_FIX_P2 = OFF_KL + 2 * T16;
constexpr int OFF_FIX_LIST = OFF_FIX_P2 + T16;  // up to 128 x 64 16-bit entries
static_assert(OFF_FIX_LIST + LT * 64 * 2 <= OFF_C0 && OFF_FIX_LIST >= OFF_TS &&
              OFF_KL % 1024 == 0, "fix-up tiles");

enum : int { B_LOAD = 0, B_OPS, B_S, B_A, B_DA, B_DAS, B_MM, B_FIX, NBAR };

__device__ __forceinline__ float2 bf2(uint32_t w) {
  return __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&w));
}

// dalpha of one (token u, channel c) with small retention, by one warp (the value is in lane 0).
// A small alpha_u (below 2^-10) leaves the suffix sum above a small remainder of terms that
// cancel, whose fp32 rounding the division magnifies.  There dalpha comes from the state
// entering u and the adjoint of Diag(alpha_u) C_{u-1}, channel c (row c), at the midpoint scale:
//   P_u = 2^{L_m} C_0 + sum_{j < u} Km_j I~_j,   Q_u = 2^{L_end - L_m} dC + sum_{t >= u} Qm_t dY_t,
//   dalpha_u = <P_u, Q_u> / alpha_u,
// where every term of P_u (u in the first half) or of Q_u (the second) carries the factor
// alpha_u, so nothing large cancels.  coef: Km of the tokens before u and Qm of those from u
// on, channel c, in fp32 (0 past T).  Tiles: 128-byte-swizzled rows of 64 bf16.
__device__ __forceinline__ float fix_up(const float* coef, const uint8_t* v, const uint8_t* dy,
                                        const uint8_t* c0, const uint8_t* dcp, int u, int c,
                                        int lane) {
  const int g4 = lane >> 3;  // tokens = g4 mod 4; the columns of 16-byte group lane & 7
  auto row16 = [&](const uint8_t* tile, int r) {
    return *reinterpret_cast<const uint4*>(
        tile + r * 128 + ((((uint32_t)lane & 7) ^ ((uint32_t)r & 7)) << 4));
  };
  auto add = [&](float (&acc)[8], float f, const uint4 x) {
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 y = bf2(w[e]);
      acc[2 * e] = fmaf(f, y.x, acc[2 * e]);
      acc[2 * e + 1] = fmaf(f, y.y, acc[2 * e + 1]);
    }
  };
  float P[8], Q[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) P[e] = Q[e] = 0.f;
#pragma unroll 4
  for (int j = g4; j < u; j += 4) add(P, coef[j], row16(v, j));
#pragma unroll 4
  for (int j = (u & ~3) + g4; j < LT; j += 4) add(Q, j >= u ? coef[j] : 0.f, row16(dy, j));
  // the four token groups' sums, the block-boundary rows, and <P_u, Q_u>
  __syncwarp();
  const uint4 c4 = row16(c0, c), e4 = row16(dcp, c);
  const uint32_t cw[4] = {c4.x, c4.y, c4.z, c4.w}, ew[4] = {e4.x, e4.y, e4.z, e4.w};
  float pq = 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 cf = bf2(cw[e]), ef = bf2(ew[e]);
#pragma unroll
    for (int h2 = 0; h2 < 2; ++h2) {
      float pe = P[2 * e + h2], qe = Q[2 * e + h2];
      pe += __shfl_xor_sync(0xffffffffu, pe, 8);
      pe += __shfl_xor_sync(0xffffffffu, pe, 16);
      qe += __shfl_xor_sync(0xffffffffu, qe, 8);
      qe += __shfl_xor_sync(0xffffffffu, qe, 16);
      pq = fmaf(pe + (h2 ? cf.y : cf.x), qe + (h2 ? ef.y : ef.x), pq);
    }
  }
  pq += __shfl_xor_sync(0xffffffffu, pq, 1);
  pq += __shfl_xor_sync(0xffffffffu, pq, 2);
  pq += __shfl_xor_sync(0xffffffffu, pq, 4);
  return pq;
}

// IN_PLACE: dalpha stands in alpha's place (a kernel of its own: the tests alone cost 1 %).
template <bool IN_PLACE>
__global__ void __launch_bounds__(kThreads, 1)
    lin_tc_bwd_kernel(const __grid_constant__ CUtensorMap tmP1,
                      const __grid_constant__ CUtensorMap tmP2,
                      const __grid_constant__ CUtensorMap tmV,
                      const __grid_constant__ CUtensorMap tmG,
                      const __grid_constant__ CUtensorMap tmA,
                      const __grid_constant__ CUtensorMap tmC0,  // states: [heads][nb][64][64]
                      const __grid_constant__ CUtensorMap tmDC,  // adjoints: [heads][nb][64][64]
                      const __grid_constant__ CUtensorMap tmDP1,
                      const __grid_constant__ CUtensorMap tmDP2,
                      const __grid_constant__ CUtensorMap tmDV, LinearProblem p, int nb) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const uint32_t sb = smem_u32(smem);
  auto bar = [&](int i) -> uint32_t { return sb + OFF_BAR + 8u * (uint32_t)i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + OFF_BAR + 96);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + OFF_BAR + 104);
  int* clamped = reinterpret_cast<int*>(smem + OFF_BAR + 108);
  int* fix_count = reinterpret_cast<int*>(smem + OFF_BAR + 112);  // small retentions found;
  int* fix_late = reinterpret_cast<int*>(smem + OFF_BAR + 116);   // entries of the late list
  float* sc = reinterpret_cast<float*>(smem + OFF_SC);
  float* s_dot = sc;             // p1_t . p2_t
  float* s_n1 = sc + LT;         // |p1_t|^2
  float* s_n2 = sc + 2 * LT;     // |p2_t|^2
  float* sum_l = sc + 3 * LT;    // [2][64] per-channel sums over the half blocks: log2 alpha
  float* sum_g = sc + 4 * LT;    // dL
  float* sum_t = sc + 5 * LT;    // Km Ys
  float* a1_s = sc + 6 * LT;     // [4][128] the groups' shares of p1_t . dq'_t
  float* a2_s = sc + 10 * LT;    // [4][128] and of p2_t . dk'_t
  float* e0_s = sc + 14 * LT;    // [64] the end term's state part
  uint16_t* fix_early = reinterpret_cast<uint16_t*>(e0_s + 64);  // [kFix] (token, channel)s

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // one 64-column split per head at d_h = 64; the heads of a block of tokens side by side
  const int tb = (int)blockIdx.x / p.H, h = (int)blockIdx.x - tb * p.H;
  const int b = tb / nb, blk = tb - b * nb, bh = b * p.H + h;
  const int t0 = blk * LT;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NBAR; ++i)
      mbar_init(bar(i), (i == B_OPS || i == B_A || i == B_DAS) ? EW : 1);
    *abort_flag = 0;
    *clamped = 0;
    *fix_count = *fix_late = 0;
    fence_mbar_init();
  }
  if (warp == W_MMA) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const Abort ab{abort_flag, p.dev_status};
  pdl_wait();

  if (warp == W_TMA) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      const uint32_t lb = bar(B_LOAD);
      mbar_arrive_expect_tx(lb, LOAD_BYTES);
      tma_load_4d(sb + OFF_P1, &tmP1, lb, 0, t0, h, b);
      tma_load_4d(sb + OFF_P2, &tmP2, lb, 0, t0, h, b);
      tma_load_4d(sb + OFF_V, &tmV, lb, 0, t0, h, b);
      tma_load_4d(sb + OFF_G, &tmG, lb, 0, t0, h, b);
      for (int k = 0; k < 2; ++k)
        tma_load_4d(sb + OFF_AL + k * LT * 128, &tmA, lb, k * 32, t0, h, b);
      tma_load_2d(sb + OFF_C0, &tmC0, lb, 0, (bh * nb + blk) * D);
      tma_load_2d(sb + OFF_DC, &tmDC, lb, 0, (bh * nb + blk) * D);
      drain_wait(lb, 0);
    }
  } else if (warp == W_MMA) {
    // ------------------------------------------------------------------ MMA issuer
    constexpr uint32_t id_s = idesc_bf16_f32(128, 128, false, false);  // S, dA
    constexpr uint32_t id_kk = idesc_bf16_f32(128, 64, false, false);  // A, B K-major
    constexpr uint32_t id_km = idesc_bf16_f32(128, 64, false, true);   // B MN-major
    constexpr uint32_t id_mm = idesc_bf16_f32(128, 64, true, true);    // A, B MN-major
    bool ok = mbar_wait_warp(bar(B_OPS), 0, ab);
    if (ok) {
      tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)  // S = Qm Km^T  (K = 64 channels)
        mma_ss_w(tmem + COL_SC, smem_desc_sw128(sb + OFF_P1 + kk * 32, 16, 1024),
                 smem_desc_sw128(sb + OFF_P2 + kk * 32, 16, 1024), id_s, kk > 0 ? 1u : 0u);
      mma_commit_w(bar(B_S));
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)  // X = G (2^{L_m} C_0)^T   (K = 64 columns n)
        mma_ss_w(tmem + COL_X, smem_desc_sw128(sb + OFF_G + kk * 32, 16, 1024),
                 smem_desc_sw128(sb + OFF_C0 + kk * 32, 16, 1024), id_kk, kk > 0 ? 1u : 0u);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)  // Ys = I~ (2^{L_end - L_m} dC)^T
        mma_ss_w(tmem + COL_YS, smem_desc_sw128(sb + OFF_V + kk * 32, 16, 1024),
                 smem_desc_sw128(sb + OFF_DCP + kk * 32, 16, 1024), id_kk, kk > 0 ? 1u : 0u);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)  // dI~ = KL dC   (A = KL [j][c], B = dC [c][n] MN-major)
        mma_ss_w(tmem + COL_DI, smem_desc_sw128(sb + OFF_KL + kk * 32, 16, 1024),
                 smem_desc_sw128(sb + OFF_DC + kk * 16 * 128, 64 * 128, 1024), id_km,
                 kk > 0 ? 1u : 0u);
      ok = mbar_wait_warp(bar(B_A), 0, ab);  // A in shared memory, S read out
    }
    if (ok) {
      tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)  // dA = G I~^T   (N = 128 tokens j, K = 64 columns)
        mma_ss_w(tmem + COL_SC, smem_desc_sw128(sb + OFF_G + kk * 32, 16, 1024),
                 smem_desc_sw128(sb + OFF_V + kk * 32, 16, 1024), id_s, kk > 0 ? 1u : 0u);
      mma_commit_w(bar(B_DA));
#pragma unroll
      for (int kk = 0; kk < LT / 16; ++kk)  // dI~ += A^T G   (A^T: MN-major view of [t][j])
        mma_ss_w(tmem + COL_DI, smem_desc_sw128(sb + OFF_AS + kk * 16 * 128, LT * 128, 1024),
                 smem_desc_sw128(sb + OFF_G + kk * 16 * 128, LT * 128, 1024), id_mm, 1u);
      ok = mbar_wait_warp(bar(B_DAS), 0, ab);  // dA in shared memory
    }
    if (ok) {
      tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < LT / 16; ++kk) {  // X += dA Km   (K = 128 tokens j)
        const uint32_t koff = (kk >> 2) * (LT * 128) + (kk & 3) * 32;
        mma_ss_w(tmem + COL_X, smem_desc_sw128(sb + OFF_DAS + koff, 16, 1024),
                 smem_desc_sw128(sb + OFF_P2 + kk * 16 * 128, LT * 128, 1024), id_km, 1u);
      }
#pragma unroll
      for (int kk = 0; kk < LT / 16; ++kk)  // Y = dA^T Qm  (K = 128 tokens t)
        mma_ss_w(tmem + COL_Y, smem_desc_sw128(sb + OFF_DAS + kk * 16 * 128, LT * 128, 1024),
                 smem_desc_sw128(sb + OFF_P1 + kk * 16 * 128, LT * 128, 1024), id_mm,
                 kk > 0 ? 1u : 0u);
    }
    mma_commit_w(bar(B_MM));  // every product (or whatever completed before an abort)
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ elementwise
    const int grp = warp >> 2;        // warpgroup
    const int t = threadIdx.x & 127;  // token of the block / TMEM lane; channel c = t & 63, half
    const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const float inv_tau_sqrt_d = 1.0f / (p.tau_s * sqrtf((float)D));
    const int c = t & 63, half = t >> 6;
    uint8_t* const p1s = smem + OFF_P1;
    uint8_t* const p2s = smem + OFF_P2;
    float* const al = reinterpret_cast<float*>(smem + OFF_AL);
    auto al_at = [&](int tok, int ch) -> float& {  // [2][128][32] fp32, 128-byte swizzle
      return al[al_swz(tok, ch)];
    };
    float* const gl = reinterpret_cast<float*>(smem + OFF_GL);  // dL [t][GS]
    float* const ts = reinterpret_cast<float*>(smem + OFF_TS);  // Km Ys [t][GS]
    bool my_clamp = false;
    bool ok = __all_sync(0xffffffffu, mbar_wait(bar(B_LOAD), 0, ab));
    // ---- log2 alpha in place of alpha (0 past T), and the (token, channel)s with a small alpha
    if (ok) {
#pragma unroll
      for (int i0 = 0; i0 < LT * D / 4; i0 += EW) {
        const int i = i0 + threadIdx.x;  // 16-byte group of the tile
        const int tok = (i >> 3) & 127;
        const bool live = t0 + tok < p.T;
        const float4 v = reinterpret_cast<const float4*>(al)[i];
        float a[4] = {v.x, v.y, v.z, v.w};
        if (live && fminf(fminf(a[0], a[1]), fminf(a[2], a[3])) < kSmallAlpha) {
          const int ch = (i >> 10) * 32 + (((i & 7) ^ (tok & 7)) << 2);
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (a[e] < kSmallAlpha) {
              const int n = atomicAdd(fix_count, 1);
              if (n < kFix) fix_early[n] = (uint16_t)(tok * 64 + ch + e);
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) a[e] = live ? log2_alpha(a[e]) : 0.f;
        reinterpret_cast<float4*>(al)[i] = make_float4(a[0], a[1], a[2], a[3]);
      }
    }
    ew_sync<NG>();
    // ---- the sums of S_t, |p1_t|, |p2_t| (groups 0, 1, 2) beside the running sums L_t in place
    // of log2 alpha (group 3: channel and half block, the second half's relative to its start)
    if (ok) {
      if (grp < 3) {
        ask_self_sums<D, 0>(p1s, p2s, t, 1 << grp, s_dot, s_n1, s_n2);
      } else {
        float lsum = 0.f;
        for (int i0 = 0; i0 < 64; i0 += 16) {
          float la[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) la[u] = al_at(half * 64 + i0 + u, c);
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            lsum += la[u];
            al_at(half * 64 + i0 + u, c) = lsum;
          }
        }
        sum_l[t] = lsum;
      }
    }
    ew_sync<NG>();
    const int n_small = *reinterpret_cast<volatile int*>(fix_count);
    const int n_early = n_small <= kFix ? n_small : 0;
    float* const coef = reinterpret_cast<float*>(smem + OFF_COEF);
    float S = 0.f, i1 = 0.f, i2 = 0.f, s1 = 0.f, s2 = 0.f;  // token t (zero past T)
    const float later = t >= 64 ? 1.f : 0.f;
    uint4 ra[2], rb[2];  // p1, p2 of token t, the group's 16 channels: Qm, Km take their place
    if (ok) {
      if (t0 + t < p.T) {
        S = 1.0f / (1.0f + __expf(-s_dot[t] * inv_tau_sqrt_d));
        i1 = rsqrtf(s_n1[t]);
        i2 = rsqrtf(s_n2[t]);
        s1 = S * i1;
        s2 = S * i2;
      }
      {
        // C_0 scaled by 2^{L_m} in place, dC scaled by 2^{L_end - L_m} into its own tile (both
        // factors <= 1): one 16-byte group of one row per thread
        const int r = threadIdx.x >> 3, k = threadIdx.x & 7;
        const float l_mid = sum_l[r], l_end = sum_l[r] + sum_l[64 + r];
        const float f0 = ex2_approx(l_mid), f1 = ex2_approx(l_end - l_mid);
        uint4* r0 = reinterpret_cast<uint4*>(smem + OFF_C0 + r * 128 + 16 * k);
        const uint4 a4 = *r0;
        const uint4 d4 = *reinterpret_cast<const uint4*>(smem + OFF_DC + r * 128 + 16 * k);
        const uint32_t aw[4] = {a4.x, a4.y, a4.z, a4.w}, dw[4] = {d4.x, d4.y, d4.z, d4.w};
        uint32_t oa[4], od[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 x = bf2(aw[e]), y = bf2(dw[e]);
          oa[e] = pack_bf16x2(x.x * f0, x.y * f0);
          od[e] = pack_bf16x2(y.x * f1, y.y * f1);
        }
        *r0 = make_uint4(oa[0], oa[1], oa[2], oa[3]);
        *reinterpret_cast<uint4*>(smem + OFF_DCP + r * 128 + 16 * k) =
            make_uint4(od[0], od[1], od[2], od[3]);
      }
      // the early fix-ups' coefficients: Km before the token, Qm from it on (each thread reads
      // the channels that it alone overwrites below)
      for (int f = 0; f < n_early; ++f) {
        const int u = fix_early[f] >> 6, ch = fix_early[f] & 63;
        if ((ch >> 4) != grp) continue;
        const float dm = dm_of(al_at(t, ch), sum_l[ch], t >= 64, my_clamp);
        const uint8_t* tile = t < u ? p2s : p1s;
        const float x = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(
            tile + t * 128 + (((ch >> 3) ^ (t & 7)) << 4) + (ch & 7) * 2));
        coef[f * LT + t] = t < u ? x * s2 * ex2_approx(-dm) : x * s1 * ex2_approx(dm);
      }
      // ---- Qm, Km in place of p1, p2, and KL: token t, the group's 16 channels
#pragma unroll
      for (int k1 = 0; k1 < 2; ++k1) {
        const int k = 2 * grp + k1;
        const uint32_t off = t * 128 + ((k ^ (t & 7)) << 4);
        ra[k1] = *reinterpret_cast<const uint4*>(p1s + off);
        rb[k1] = *reinterpret_cast<const uint4*>(p2s + off);
        const uint32_t aw[4] = {ra[k1].x, ra[k1].y, ra[k1].z, ra[k1].w};
        const uint32_t bw[4] = {rb[k1].x, rb[k1].y, rb[k1].z, rb[k1].w};
        uint32_t qm[4], km[4], kl[4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {  // four channels
          const float4 L4 = *reinterpret_cast<const float4*>(&al_at(t, 8 * k + 4 * q));
          const float4 M4 = *reinterpret_cast<const float4*>(sum_l + 8 * k + 4 * q);
          const float4 E4 = *reinterpret_cast<const float4*>(sum_l + 64 + 8 * k + 4 * q);
          const float Lv[4] = {L4.x, L4.y, L4.z, L4.w}, Mv[4] = {M4.x, M4.y, M4.z, M4.w};
          const float Ev[4] = {E4.x, E4.y, E4.z, E4.w};
          float Lt[4], dm[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            Lt[j] = fmaf(Mv[j], later, Lv[j]);
            dm[j] = Lt[j] - Mv[j];
          }
          clamp_exponents(dm, my_clamp);
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float2 x = bf2(aw[2 * q + e]), y = bf2(bw[2 * q + e]);
            float r[2][3];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int j = 2 * e + u;
              const float xs = (u ? x.y : x.x) * s1, ys = (u ? y.y : y.x) * s2;
              r[u][0] = xs * ex2_approx(dm[j]);
              r[u][1] = ys * ex2_approx(-dm[j]);
              r[u][2] = ys * ex2_approx((Mv[j] + Ev[j]) - Lt[j]);  // KL (factor <= 1)
            }
            qm[2 * q + e] = pack_bf16x2(r[0][0], r[1][0]);
            km[2 * q + e] = pack_bf16x2(r[0][1], r[1][1]);
            kl[2 * q + e] = pack_bf16x2(r[0][2], r[1][2]);
          }
        }
        *reinterpret_cast<uint4*>(p1s + off) = make_uint4(qm[0], qm[1], qm[2], qm[3]);
        *reinterpret_cast<uint4*>(p2s + off) = make_uint4(km[0], km[1], km[2], km[3]);
        *reinterpret_cast<uint4*>(smem + OFF_KL + off) = make_uint4(kl[0], kl[1], kl[2], kl[3]);
      }
      fence_async_smem();
      mbar_arrive(bar(B_OPS));
    }
    // ---- A = tril(S, -1), then dA = tril(G I~^T, -1), as bf16 rows [t][j] in shared memory
    // (the products read them K-major and, transposed, MN-major): 32 columns per group
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(pass == 0 ? B_S : B_DA), 0, ab));
      if (!ok) break;
      tc_fence_after();
      uint8_t* dst = smem + (pass == 0 ? OFF_AS : OFF_DAS);
      const int c0 = 32 * grp;
      uint32_t pk[16];
      if (grp <= (warp & 3)) {  // some column of the warp's rows is unmasked
        uint32_t s[32];
        tmem_ld32(trow + COL_SC + c0, s);
        tmem_ld_wait();
        if (grp == (warp & 3)) {  // the warp's diagonal square
#pragma unroll
          for (int j = 0; j < 32; ++j) s[j] = c0 + j < t ? s[j] : 0u;
        }
#pragma unroll
        for (int j = 0; j < 32; j += 2)
          pk[j >> 1] = pack_bf16x2(__uint_as_float(s[j]), __uint_as_float(s[j + 1]));
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) pk[j] = 0u;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4*>(dst + swz(t, c0 + 8 * q, LT)) =
            make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
      fence_async_smem();
      tc_fence_before();
      mbar_arrive(bar(pass == 0 ? B_A : B_DAS));
    }
    // ---- the few small retentions' dalpha while the products run (dY, I~ and the state tiles
    // still stand), a warp each
    if (n_early > 0) {
      ew_sync<NG>();  // the coefficients and the scaled state tiles are written
      if (ok && warp < n_early) {
        const int u = fix_early[warp] >> 6, ch = fix_early[warp] & 63;
        const long long at =
            (long long)b * p.sB + (long long)h * p.sH + (long long)(t0 + u) * p.sT + ch;
        const float a = __ldg(p.alpha + at);
        const float pq = fix_up(coef + warp * LT, smem + OFF_V, smem + OFF_G, smem + OFF_C0,
                                smem + OFF_DCP, u, ch, lane);
        if (IN_PLACE) __syncwarp();  // kept, in place of the warp's coefficients, until every alpha
                                     // of the block has been read
        if (lane == 0) *(IN_PLACE ? coef + warp * LT : p.dalpha + at) = pq / a;
      }
      ew_sync<NG>();  // dY has been read: dv takes its place
    }
    // ---- every product done: token t, the group's channels
    ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(B_MM), 0, ab));
    uint8_t* const gs = smem + OFF_G;
    float dq[16], dk[16];
    if (ok) {
      tc_fence_after();
      // dq' = 2^{L_t - L_m} X, dk' = 2^{L_m - L_t} Y (Y = dA^T Qm + Ys), the group's shares of
      // p1 . dq' and p2 . dk', dL = Qm X - Km Y and Km Ys (Qm, Km as the products read them),
      // dv = dI~ + dY (in dY's place)
      float A1 = 0.f, A2 = 0.f;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int kc = 2 * grp + k;
        uint32_t x[8], y[8], ys[8], di[8];
        tmem_ld8(trow + COL_X + 8 * kc, x);
        tmem_ld8(trow + COL_Y + 8 * kc, y);
        tmem_ld8(trow + COL_YS + 8 * kc, ys);
        tmem_ld8(trow + COL_DI + 8 * kc, di);
        tmem_ld_wait();
        const uint32_t off = t * 128 + ((kc ^ (t & 7)) << 4);
        const uint4 a4 = ra[k], b4 = rb[k];
        const uint4 m4 = *reinterpret_cast<const uint4*>(p1s + off);  // Qm, Km as the products
        const uint4 n4 = *reinterpret_cast<const uint4*>(p2s + off);  // read them
        const uint4 g4 = *reinterpret_cast<const uint4*>(gs + off);
        const float4 M0 = *reinterpret_cast<const float4*>(sum_l + 8 * kc);
        const float4 M1 = *reinterpret_cast<const float4*>(sum_l + 8 * kc + 4);
        const float Mv[8] = {M0.x, M0.y, M0.z, M0.w, M1.x, M1.y, M1.z, M1.w};
        const uint32_t mw[4] = {m4.x, m4.y, m4.z, m4.w}, nw[4] = {n4.x, n4.y, n4.z, n4.w};
        const float4 L0 = *reinterpret_cast<const float4*>(&al_at(t, 8 * kc));
        const float4 L1 = *reinterpret_cast<const float4*>(&al_at(t, 8 * kc + 4));
        const float Lv[8] = {L0.x, L0.y, L0.z, L0.w, L1.x, L1.y, L1.z, L1.w};
        const uint32_t aw[4] = {a4.x, a4.y, a4.z, a4.w}, bw[4] = {b4.x, b4.y, b4.z, b4.w},
                       gw[4] = {g4.x, g4.y, g4.z, g4.w};
        float dl[8], tv[8];
        uint32_t dvw[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 xa = bf2(aw[e]), yb = bf2(bw[e]), g = bf2(gw[e]);
          const float2 qm2 = bf2(mw[e]), km2 = bf2(nw[e]);
          float dvv[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int i = 2 * e + u, j = 8 * k + i;
            const float pv = u ? xa.y : xa.x, kv = u ? yb.y : yb.x;
            const float qm = u ? qm2.y : qm2.x, km = u ? km2.y : km2.x;
            const float X = __uint_as_float(x[i]), Ysv = __uint_as_float(ys[i]);
            const float Y = __uint_as_float(y[i]) + Ysv;
            const float dm = clamp_exponent(fmaf(Mv[i], later, Lv[i]) - Mv[i]);
            dq[j] = ex2_approx(dm) * X;
            dk[j] = ex2_approx(-dm) * Y;
            A1 = fmaf(pv, dq[j], A1);
            A2 = fmaf(kv, dk[j], A2);
            dl[2 * e + u] = qm * X - km * Y;
            tv[2 * e + u] = km * Ysv;
            dvv[u] = __uint_as_float(di[i]) + (u ? g.y : g.x);
          }
          dvw[e] = pack_bf16x2(dvv[0], dvv[1]);
        }
        *reinterpret_cast<uint4*>(gs + off) = make_uint4(dvw[0], dvw[1], dvw[2], dvw[3]);
        float* gr = gl + t * GS + 8 * kc;
        *reinterpret_cast<float4*>(gr) = make_float4(dl[0], dl[1], dl[2], dl[3]);
        *reinterpret_cast<float4*>(gr + 4) = make_float4(dl[4], dl[5], dl[6], dl[7]);
        float* tr = ts + t * GS + 8 * kc;
        *reinterpret_cast<float4*>(tr) = make_float4(tv[0], tv[1], tv[2], tv[3]);
        *reinterpret_cast<float4*>(tr + 4) = make_float4(tv[4], tv[5], tv[6], tv[7]);
      }
      a1_s[grp * 128 + t] = A1;
      a2_s[grp * 128 + t] = A2;
    }
    // dalpha's division reads alpha again, rows of 16 threads (in flight during the sums)
    const long long abase = (long long)b * p.sB + (long long)h * p.sH + 4 * (threadIdx.x & 15);
    const int arow = threadIdx.x >> 4;  // rows arow + 32 i
    float4 av[4];
    ew_sync<NG>();
    if (ok) {
      // through S_t and the normalisation of p1, p2 (written in their place)
      //   dp1 = S/|p1| dq' - S/|p1|^3 (p1 . dq') p1 + du p2, and symmetrically dp2,
      //   du = (p1 . dq' / |p1| + p2 . dk' / |p2|) S (1 - S) / (tau_S sqrt(d_h))
      const float A1 = ((a1_s[t] + a1_s[128 + t]) + a1_s[256 + t]) + a1_s[384 + t];
      const float A2 = ((a2_s[t] + a2_s[128 + t]) + a2_s[256 + t]) + a2_s[384 + t];
      const float du = (i1 * A1 + i2 * A2) * S * (1.0f - S) * inv_tau_sqrt_d;
      const float c1 = s1 * i1 * i1 * A1, c2 = s2 * i2 * i2 * A2;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const uint32_t off = t * 128 + (((2 * grp + k) ^ (t & 7)) << 4);
        const uint4 a4 = ra[k], b4 = rb[k];
        const uint32_t aw[4] = {a4.x, a4.y, a4.z, a4.w}, bw[4] = {b4.x, b4.y, b4.z, b4.w};
        uint32_t o1[4], o2[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 xa = bf2(aw[e]), yb = bf2(bw[e]);
          float r1v[2], r2v[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int j = 8 * k + 2 * e + u;
            const float pv = u ? xa.y : xa.x, kv = u ? yb.y : yb.x;
            r1v[u] = fmaf(s1, dq[j], fmaf(-c1, pv, du * kv));
            r2v[u] = fmaf(s2, dk[j], fmaf(-c2, kv, du * pv));
          }
          o1[e] = pack_bf16x2(r1v[0], r1v[1]);
          o2[e] = pack_bf16x2(r2v[0], r2v[1]);
        }
        *reinterpret_cast<uint4*>(p1s + off) = make_uint4(o1[0], o1[1], o1[2], o1[3]);
        *reinterpret_cast<uint4*>(p2s + off) = make_uint4(o2[0], o2[1], o2[2], o2[3]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int tok = t0 + arow + 32 * i;
        av[i] = make_float4(1.f, 1.f, 1.f, 1.f);
        if (tok < p.T)
          av[i] = __ldg(reinterpret_cast<const float4*>(p.alpha + abase + (long long)tok * p.sT));
      }
      fence_async_smem();
      // ---- per channel and half block: the sums of dL (group 0) and of Km Ys (group 1); per
      // channel (group 2) end's state part, sum_n (2^{L_m} C_0)[c][n] (2^{L_end - L_m} dC)[c][n]
      if (grp < 2) {
        const float* src = (grp == 0 ? gl : ts) + half * 64 * GS + c;
        float sum = 0.f;
#pragma unroll
        for (int i0 = 0; i0 < 64; i0 += 16) {  // 16 independent loads in flight
          float v16[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) v16[u] = src[(i0 + u) * GS];
#pragma unroll
          for (int u = 0; u < 16; ++u) sum += v16[u];
        }
        (grp == 0 ? sum_g : sum_t)[t] = sum;
      } else if (grp == 2 && half == 0) {
        float e0 = 0.f;
        const uint8_t* rc0 = smem + OFF_C0 + c * 128;
        const uint8_t* rdp = smem + OFF_DCP + c * 128;
#pragma unroll
        for (int k0 = 0; k0 < 8; ++k0) {  // same swizzle in both tiles: a plain row dot
          const int k = (k0 + c) & 7;     // rows 128 bytes apart: rotate the 16-byte groups
          const uint4 a4 = *reinterpret_cast<const uint4*>(rc0 + 16 * k);
          const uint4 d4 = *reinterpret_cast<const uint4*>(rdp + 16 * k);
          const uint32_t aw[4] = {a4.x, a4.y, a4.z, a4.w}, dw[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 x = bf2(aw[e]), y = bf2(dw[e]);
            e0 = fmaf(x.x, y.x, fmaf(x.y, y.y, e0));
          }
        }
        e0_s[c] = e0;
      }
    }
    ew_sync<NG>();
    if (ok && grp == 0) {
      // the suffix sums end + sum_{t >= u} dL_t in dL's place; what the block's end and (for the
      // first half) the later half carry comes first
      float run = e0_s[c] + sum_t[c] + sum_t[64 + c] + (half == 0 ? sum_g[64 + c] : 0.f);
      float* col = gl + half * 64 * GS + c;
#pragma unroll
      for (int i0 = 48; i0 >= 0; i0 -= 16) {
        float g16[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) g16[u] = col[(i0 + u) * GS];
#pragma unroll
        for (int u = 15; u >= 0; --u) {
          run += g16[u];
          col[(i0 + u) * GS] = run;
        }
      }
    } else if (ok && grp == 1 && lane == 0) {  // 32 rows of dp1, dp2, dv per warp
      const int r0 = (warp & 3) * 32;
      if (t0 + r0 < p.T) {
        const uint32_t so = (uint32_t)r0 * 128;
        tma_store_4d(&tmDP1, sb + OFF_P1 + so, 0, t0 + r0, h, b);
        tma_store_4d(&tmDP2, sb + OFF_P2 + so, 0, t0 + r0, h, b);
        tma_store_4d(&tmDV, sb + OFF_G + so, 0, t0 + r0, h, b);
        tma_store_commit();
      }
    }
    ew_sync<NG>();
    // ---- dalpha_u = (end + sum_{t >= u} dL_t) / alpha_u, rows of 16 threads, but for small
    // alphas: those were written above or are listed for the late fix-up
    uint16_t* const late_list = reinterpret_cast<uint16_t*>(smem + OFF_FIX_LIST);
    if (ok) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int tok = arow + 32 * i;
        const float4 r4 = *reinterpret_cast<const float4*>(gl + tok * GS + 4 * (threadIdx.x & 15));
        const float a[4] = {av[i].x, av[i].y, av[i].z, av[i].w};
        const float d[4] = {r4.x / a[0], r4.y / a[1], r4.z / a[2], r4.w / a[3]};
        float* const to = p.dalpha + abase + (long long)(t0 + tok) * p.sT;
        if (t0 + tok >= p.T) continue;
        if (!(fminf(fminf(a[0], a[1]), fminf(a[2], a[3])) < kSmallAlpha)) {
          *reinterpret_cast<float4*>(to) = make_float4(d[0], d[1], d[2], d[3]);
          continue;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (!(a[e] < kSmallAlpha))
            to[e] = d[e];
          else if (n_early == 0)
            late_list[atomicAdd(fix_late, 1)] =
                (uint16_t)(tok * 64 + 4 * (threadIdx.x & 15) + e);
        }
      }
    }
    if (n_small > n_early) {  // more than kFix: their tiles again, a warp per (token, channel)
      ew_sync<NG>();
      const int n_late = *reinterpret_cast<volatile int*>(fix_late);
      if (ok && threadIdx.x == 0) {
        fence_async_smem();  // the dL arrays' generic accesses precede the copies
        mbar_arrive_expect_tx(bar(B_FIX), 3 * T16);
        tma_load_4d(sb + OFF_FIX_G, &tmG, bar(B_FIX), 0, t0, h, b);
        tma_load_4d(sb + OFF_FIX_P1, &tmP1, bar(B_FIX), 0, t0, h, b);
        tma_load_4d(sb + OFF_FIX_P2, &tmP2, bar(B_FIX), 0, t0, h, b);
      }
      ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(B_FIX), 0, ab));
      for (int f = warp; ok && f < n_late; f += NG * 4) {
        const int u = late_list[f] >> 6, ch = late_list[f] & 63;
        bool unused_clamp = false;
        float* const cf = coef + warp * LT;
        for (int tok = lane; tok < LT; tok += 32) {
          float x = 0.f;
          if (t0 + tok < p.T) {
            const float St = 1.0f / (1.0f + __expf(-s_dot[tok] * inv_tau_sqrt_d));
            const float dm = dm_of(al_at(tok, ch), sum_l[ch], tok >= 64, unused_clamp);
            x = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(
                smem + (tok < u ? OFF_FIX_P2 : OFF_FIX_P1) + tok * 128 +
                (((ch >> 3) ^ (tok & 7)) << 4) + (ch & 7) * 2));
            x = tok < u ? x * (St * rsqrtf(s_n2[tok])) * ex2_approx(-dm)
                        : x * (St * rsqrtf(s_n1[tok])) * ex2_approx(dm);
          }
          cf[tok] = x;
        }
        __syncwarp();
        const float pq = fix_up(cf, smem + OFF_V, smem + OFF_FIX_G, smem + OFF_C0,
                                smem + OFF_DCP, u, ch, lane);
        const long long at =
            (long long)b * p.sB + (long long)h * p.sH + (long long)(t0 + u) * p.sT + ch;
        if (lane == 0) p.dalpha[at] = pq / __ldg(p.alpha + at);
        __syncwarp();
      }
    }
    if (IN_PLACE && ok && warp < n_early && lane == 0) {
      const int u = fix_early[warp] >> 6, ch = fix_early[warp] & 63;
      p.dalpha[(long long)b * p.sB + (long long)h * p.sH + (long long)(t0 + u) * p.sT + ch] =
          coef[warp * LT];
    }
    if (lane == 0) tma_store_wait_read_all();
    if (my_clamp) atomicExch(clamped, 1);
  }

  if (warp == W_MMA) drain_wait(bar(B_MM), 0);  // no product in flight past the teardown
  if (threadIdx.x == 0 && *fix_late > 0) drain_wait(bar(B_FIX), 0);  // nor the fix-up's copies
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *clamped && p.dev_status && !*abort_flag)
    atomicExch(p.dev_status, (int)RELATION_ERR_UNSUPPORTED);
  if (warp == W_MMA) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace bwd
}  // namespace lintc

bool linear_tc_bwd_supports(const LinearProblem& p) {
  return p.dtype == RELATION_BF16 && p.d == 64 && p.sB % 8 == 0 && p.sT % 8 == 0 &&
         p.sH % 8 == 0;
}

size_t linear_tc_bwd_workspace_bytes(const LinearProblem& p) {
  if (!linear_tc_bwd_supports(p)) return 0;
  const long long heads = (long long)p.B * p.H, nb = (p.T + lintc::LT - 1) / lintc::LT;
  return lintc::bwd_bytes(heads, nb, 64, nullptr, nullptr);
}

// Three launches: the two state passes (launch_states), then one CTA per (head, block).
cudaError_t launch_linear_tc_bwd(const LinearProblem& p, cudaStream_t s) {
  using namespace lintc;
  if (!linear_tc_bwd_supports(p) || !p.workspace) return cudaErrorInvalidValue;
  const int nb = (p.T + LT - 1) / LT;
  const long long heads = (long long)p.B * p.H;
  const long long grid = heads * nb;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  cudaError_t e;
  auto* const kernel = p.dalpha == p.alpha ? bwd::lin_tc_bwd_kernel<true> : bwd::lin_tc_bwd_kernel<false>;
  if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                bwd::SMEM)) != cudaSuccess) {
    note_failure("linear chunked backward: shared memory attribute");
    return e;
  }
  if ((e = launch_states(p, p.dy, p.workspace, s)) != cudaSuccess) return e;
  LinCp cp{};
  bwd_bytes(heads, nb, 64, &cp, p.workspace);
  Problem q{};  // the bf16 tensor-map helper's view of the shapes
  q.B = p.B; q.T = p.T; q.H = p.H; q.d = p.d;
  q.sB = p.sB; q.sT = p.sT; q.sH = p.sH;
  CUtensorMap m1, m2, mv, mg, ma, mc0, mdc, o1, o2, ov;
  if (!tc::make_tmap_bf16(&m1, p.p1, q, LT) || !tc::make_tmap_bf16(&m2, p.p2, q, LT) ||
      !tc::make_tmap_bf16(&mv, p.v, q, LT) || !tc::make_tmap_bf16(&mg, p.dy, q, LT) ||
      !make_tmap_alpha(&ma, p, true) || !make_tmap_c0(&mc0, cp.dC, heads * nb * 64, 64) ||
      !make_tmap_c0(&mdc, cp.dQ, heads * nb * 64, 64) || !tc::make_tmap_bf16(&o1, p.dp1, q, 32) ||
      !tc::make_tmap_bf16(&o2, p.dp2, q, 32) || !tc::make_tmap_bf16(&ov, p.dv, q, 32)) {
    note_failure("linear chunked backward: TMA descriptors");
    return cudaErrorInvalidValue;
  }
  e = launch_pdl(kernel, dim3((unsigned)grid), bwd::kThreads, bwd::SMEM, s, 1, m1, m2,
                 mv, mg, ma, mc0, mdc, o1, o2, ov, p, nb);
  if (e != cudaSuccess) note_failure("linear chunked backward: launch");
  return e;
}

}  // namespace rel
