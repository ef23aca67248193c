// relation_linear_tc.cu -- chunked tensor-core form of the Linear Relation forward
// (Sec. 5.2, Eq. (decayed-relation-state); App. A.4), bf16, d_h 64 or 128.
//
// The recurrence (relation_linear.cu) regrouped into blocks of LT = 128 tokens.  Per head,
// with q'_t = S_t ^p1_t, k'_t = S_t ^p2_t (Ask Self folded into the unit coordinates), the
// channel-wise cumulative log-retention inside a block L_t = sum_{u <= t} log2 alpha_u
// (a_t = 2^{L_t}), and C_0 the state the block starts from (fp32, d x d, kept in TMEM):
//   E_t = (a_t q'_t)^T C_0 + sum_{j < t} (q'_t . (a_t / a_j) k'_j) I~_j,   Y_t = I~_t + E_t
//   C_L = Diag(a_L) C_0 + sum_j ((a_L / a_j) k'_j) I~_j^T
// so that a block is four tcgen05 products:
//   S   = Qm Km^T          Qm_t = q'_t 2^{L_t - L_m}, Km_j = k'_j 2^{L_m - L_j}   (M = N = 128)
//   E   = Qs C_0           Qs_t = q'_t 2^{L_t}
//   E  += tril(S, -1) I~   (S masked and packed to bf16 in TMEM: a TS product)
//   C  <- Diag(2^{L_L}) C + KL^T I~,   KL_j = k'_j 2^{L_L - L_j}
// The ratio a_t / a_j of the intra-block pairs is split at the block's midpoint m (the
// 64th token), so each factor covers at most half a block of decay; the inter-block and
// state factors are at most 1.  A factor beyond 2^120 (a channel decaying below 2^-120
// within 64 tokens) is clamped and the call reports RELATION_ERR_UNSUPPORTED through
// dev_status: the result is then not exact (the recurrent kernels have no such limit).
//
// One CTA per (head, 64 information columns): the columns of C and Y never mix, so a
// d_h = 128 head runs as two CTAs that share the Q / K operands' arithmetic.  Elementwise
// warpgroups of four warps (thread = token, or TMEM lane; the groups split the channels or
// columns), then a warp that issues the TMA loads and one (warp-uniform, elect.sync) the
// MMAs.  The block is a chain of short phases around small products: neither HBM nor a pipe
// bounds it but the latency of those phases, so their work is spread over as many warps as
// the SM holds: four groups on the sequential walk (one CTA per SM, its next block's loads
// in flight), two on the one-block modes at d_h = 64, which leave room for a second CTA per SM
// whose phases fill this one's waits.  With one group (one CTA per SM) the sequential walk took
// 126 us at B 8, H 12, T 2048, d 64; four groups 93; with the logarithms on every warp, the next
// block's sums taken while the output product runs and the stores on the TMA warp 82.  At B 1,
// H 12, T 32768 DELTA, the scan and OUT took 140, 27 and 177 us, now 78, 16 and 95.
// Every mbarrier wait is bounded (common.cuh); a warp whose wait gave up keeps
// meeting the warpgroups' barriers and skips the work between them.
#include <cudaTypedefs.h>
#include <math.h>

#include "relation_linear_tc.cuh"

namespace rel {
namespace lintc {
template <int D, int MODE>
struct Cfg {
  static constexpr bool SEQ = MODE == MODE_SEQ;
  static constexpr bool DELTA = MODE == MODE_DELTA || MODE == MODE_BOTH;
  static constexpr int NG = (D == 64 && !SEQ) ? 2 : 4;  // elementwise warpgroups
  static constexpr int CTAS = (D == 64 && !SEQ) ? 2 : 1;  // per SM
  static constexpr int EW = NG * 128, W_TMA = NG * 4, W_MMA = W_TMA + 1;
  static constexpr int THREADS = EW + 64;
  static constexpr int KB = D / 64;          // 64-channel (128-byte) blocks of a p tile
  static constexpr int PT = LT * D * 2;      // p1 / p2 / operand tile, [128 t][D] bf16
  static constexpr int VT = LT * NC * 2;     // the CTA's 64 columns of I~
  static constexpr int AT = LT * D * 4;      // alpha, [D / 32][128 t][32] fp32
  static constexpr int C0T = D * NC * 2;     // bf16 copy of C_0's 64 columns, [D c][64 n]
  // Input stages (SEQ at d_h = 64: the next block's loads overlap the current block): p2 (then
  // Km in place; DELTA: KL), p1 (then Qm in place, then the Y staging; BOTH: Qs), the CTA's I~
  // columns, dY (BOTH), alpha (then its running log2 sums).
  static constexpr int STAGES = (D == 64 && SEQ) ? 2 : 1;
  static constexpr int OFF_P2 = 0;
  static constexpr int OFF_P1 = OFF_P2 + PT;
  static constexpr int OFF_V = OFF_P1 + PT;
  static constexpr int OFF_G = OFF_V + VT;
  static constexpr int OFF_A = OFF_G + (MODE == MODE_BOTH ? VT : 0);
  static constexpr int STAGE = OFF_A + AT;
  // KL as the state product's A operand has 128 channels: at d_h = 64 the tile after it (Qs,
  // p1) takes the upper 64, whose result rows are read by nobody (BOTH: they are Qs^T dY)
  static constexpr int OFF_KL = DELTA ? OFF_P2 : STAGES * STAGE;
  static constexpr int OFF_QS = SEQ ? OFF_KL + PT : STAGES * STAGE;
  static constexpr int OFF_C0 = SEQ ? OFF_QS + PT : (DELTA ? STAGE : OFF_QS + PT);
  // the per-token / per-channel scalars; AHEAD: two sets, the next block's sums are taken while
  // the current block's output product runs.  d_h = 128 SEQ has no room: they stand in the C0
  // tile before the copy is written there
  static constexpr bool AHEAD = STAGES == 2, IN_C0 = SEQ && D == 128;
  static constexpr int OFF_SC = IN_C0 || DELTA ? OFF_C0 : OFF_C0 + C0T;
  static constexpr int SCB = 5 * LT * 4;
  static constexpr int OFF_BAR = IN_C0 ? OFF_C0 + C0T : OFF_SC + (AHEAD ? 2 : 1) * SCB;
  static constexpr int SMEM = OFF_BAR + 128 + 1024;
  static constexpr uint32_t LOAD_BYTES =
      2 * PT + VT + AT + (MODE == MODE_OUT ? C0T : 0) + (MODE == MODE_BOTH ? VT : 0);
  // TMEM columns: S 128 | E 64 | P 64 (S masked, bf16) | C 64; DELTA: C 64 (BOTH: 128) alone
  static constexpr int COL_S = 0, COL_E = 128, COL_P = 192, COL_C = DELTA ? 0 : 256;
  static constexpr int TMEM = SEQ ? 512 : (DELTA ? 128 : 256);
  static_assert(SCB <= C0T, "scalars in the C0 tile");
  static_assert(CTAS * (SMEM + 1024) <= 233472, "shared memory");
};

// 32 bytes to global memory (one sector)
__device__ __forceinline__ void st_global_32(float* p, const uint32_t* r) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

template <int D, int MODE>
__global__ void __launch_bounds__(Cfg<D, MODE>::THREADS, Cfg<D, MODE>::CTAS)
    lin_tc_fwd_kernel(const __grid_constant__ CUtensorMap tmP1,
                      const __grid_constant__ CUtensorMap tmP2,
                      const __grid_constant__ CUtensorMap tmV,
                      const __grid_constant__ CUtensorMap tmG,
                      const __grid_constant__ CUtensorMap tmA,
                      const __grid_constant__ CUtensorMap tmY,
                      const __grid_constant__ CUtensorMap tmC0, LinearProblem p, LinCp cp) {
  using C = Cfg<D, MODE>;
  constexpr bool SEQ = C::SEQ, DELTA = C::DELTA, BOTH = MODE == MODE_BOTH;
  constexpr int NG = C::NG;
  static_assert(!BOTH || D == 64, "both contributions in one product: d_h = 64");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const uint32_t sb = smem_u32(smem);
  auto bar = [&](int i) -> uint32_t { return sb + C::OFF_BAR + 8u * (uint32_t)i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_BAR + 96);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_BAR + 104);
  int* clamped = reinterpret_cast<int*>(smem + C::OFF_BAR + 108);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int NSPLIT = D / NC;
  const int nb = (p.T + LT - 1) / LT;
  // SEQ: one CTA per (head, split) over blocks [0, nb); DELTA / BOTH / OUT: one block per CTA
  const int cta_blk = SEQ ? 0 : (int)(blockIdx.x % nb);
  const int bhs = SEQ ? (int)blockIdx.x : (int)(blockIdx.x / nb);
  const int split = bhs % NSPLIT;
  const int bh = bhs / NSPLIT;
  const int b = bh / p.H, h = bh % p.H;
  const int blk_first = cta_blk, blk_end = SEQ ? nb : cta_blk + 1;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NBAR; ++i)  // arrivals of the elementwise threads, or one
      mbar_init(bar(i), (i == B_OPS || i == B_C0 || i == B_A || i == B_EPI || i == B_EPI + 1)
                            ? C::EW : 1);
    *abort_flag = 0;
    *clamped = 0;
    fence_mbar_init();
  }
  if (warp == C::W_MMA) tmem_alloc(smem_u32(tmem_slot), C::TMEM);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const Abort ab{abort_flag, p.dev_status};

  if (warp == C::W_TMA) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      // Y of block it (staged in its p1 tile) by TMA, once every elementwise thread has
      // written its part and read the stage's I~
      auto store_y = [&](int it) -> bool {
        const int st = it % C::STAGES;
        if (!mbar_wait(bar(B_EPI + st), (it / C::STAGES) & 1, ab)) return false;
        for (int q = 0; q < LT && (blk_first + it) * LT + q < p.T; q += 32)
          tma_store_4d(&tmY, sb + st * C::STAGE + C::OFF_P1 + q * 128, split * NC,
                       (blk_first + it) * LT + q, h, b);
        tma_store_commit();
        tma_store_wait_read_all();  // before the stage is loaded again (or the CTA exits)
        return true;
      };
      const int n_it = blk_end - blk_first;
      int issued = 0;
      bool ok = true;
      for (int blk = blk_first; blk < blk_end; ++blk) {
        const int it = blk - blk_first;
        const int st = it % C::STAGES, use = it / C::STAGES;
        // the stage's previous block: its MMAs are done and its output is stored
        if (use > 0 && (!(ok = store_y(it - C::STAGES)) ||
                        !(ok = mbar_wait(bar(B_FREE + st), (use - 1) & 1, ab))))
          break;
        const int t0 = blk * LT;
        const uint32_t sg = sb + st * C::STAGE;
        const uint32_t lb = bar(B_LOAD + st);
        mbar_arrive_expect_tx(lb, C::LOAD_BYTES);
        for (int kb = 0; kb < C::KB; ++kb) {
          tma_load_4d(sg + C::OFF_P1 + kb * LT * 128, &tmP1, lb, kb * 64, t0, h, b);
          tma_load_4d(sg + C::OFF_P2 + kb * LT * 128, &tmP2, lb, kb * 64, t0, h, b);
        }
        for (int k = 0; k < D / 32; ++k)
          tma_load_4d(sg + C::OFF_A + k * LT * 128, &tmA, lb, k * 32, t0, h, b);
        tma_load_4d(sg + C::OFF_V, &tmV, lb, split * NC, t0, h, b);
        if (BOTH) tma_load_4d(sg + C::OFF_G, &tmG, lb, split * NC, t0, h, b);
        if (MODE == MODE_OUT)  // the state the block starts from, in the MN-major B layout
          tma_load_2d(sb + C::OFF_C0, &tmC0, lb, 0, (bhs * nb + blk) * D);
        issued = it + 1;
      }
      if (!DELTA)
        for (int it = max(0, n_it - C::STAGES); ok && it < n_it; ++it) ok = store_y(it);
      if (ab.raised())  // copies in flight land before the CTA releases its shared memory
        for (int it = issued - C::STAGES > 0 ? issued - C::STAGES : 0; it < issued; ++it)
          drain_wait(bar(B_LOAD + it % C::STAGES), (it / C::STAGES) & 1);
    }
  } else if (warp == C::W_MMA) {
    // ------------------------------------------------------------------ MMA issuer
    constexpr uint32_t id_s = idesc_bf16_f32(128, 128, false, false);
    constexpr uint32_t id_e = idesc_bf16_f32(128, NC, false, true);
    constexpr uint32_t id_c = idesc_bf16_f32(128, BOTH ? 2 * NC : NC, true, true);
    bool ok = true;
    for (int blk = blk_first; ok && blk < blk_end; ++blk) {
      const int it = blk - blk_first;
      const uint32_t ph = it & 1;
      const int st = it % C::STAGES;
      const uint32_t sg = sb + st * C::STAGE;
      if (!(ok = mbar_wait_warp(bar(B_OPS), ph, ab))) break;
      tc_fence_after();
      if (!DELTA) {
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {  // S = Qm Km^T
          const uint32_t koff = (kk >> 2) * (LT * 128) + (kk & 3) * 32;
          mma_ss_w(tmem + C::COL_S, smem_desc_sw128(sg + C::OFF_P1 + koff, 16, 1024),
                   smem_desc_sw128(sg + C::OFF_P2 + koff, 16, 1024), id_s, kk > 0 ? 1u : 0u);
        }
        mma_commit_w(bar(B_S));
        if (SEQ) {  // (OUT: C0 came with the block's inputs)
          if (!(ok = mbar_wait_warp(bar(B_C0), ph, ab))) break;
          tc_fence_after();
        }
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {  // E = Qs C_0
          const uint32_t koff = (kk >> 2) * (LT * 128) + (kk & 3) * 32;
          mma_ss_w(tmem + C::COL_E, smem_desc_sw128(sb + C::OFF_QS + koff, 16, 1024),
                   smem_desc_sw128(sb + C::OFF_C0 + kk * 16 * 128, D * 128, 1024), id_e,
                   kk > 0 ? 1u : 0u);
        }
        if (!(ok = mbar_wait_warp(bar(B_A), ph, ab))) break;
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < LT / 16; ++kk)  // E += tril(S, -1) I~   (A from TMEM)
          mma_ts_w(tmem + C::COL_E, tmem + C::COL_P + kk * 8,
                   smem_desc_sw128(sg + C::OFF_V + kk * 16 * 128, LT * 128, 1024), id_e, 1u);
        mma_commit_w(bar(B_E));
      }
      if (MODE != MODE_OUT) {
        // SEQ: C += KL^T I~ (C decayed by the threads); DELTA: the block's own sum; BOTH:
        // [KL | Qs]^T [I~ | dY], whose diagonal quarters are the two contributions
#pragma unroll
        for (int kk = 0; kk < LT / 16; ++kk)
          mma_ss_w(tmem + C::COL_C,
                   smem_desc_sw128(sb + C::OFF_KL + kk * 16 * 128, LT * 128, 1024),
                   smem_desc_sw128(sg + C::OFF_V + kk * 16 * 128, LT * 128, 1024), id_c,
                   ((SEQ && blk > 0) || kk > 0) ? 1u : 0u);
        mma_commit_w(bar(B_STATE));
      }
      if (SEQ) mma_commit_w(bar(B_FREE + st));
    }
    // SEQ: the last commits land before the CTA exits (EW warps have waited for the others)
    if (SEQ && ok)
      for (int it = max(0, nb - C::STAGES); it < nb; ++it)
        mbar_wait_warp(bar(B_FREE + it % C::STAGES), (it / C::STAGES) & 1, ab);
    __syncwarp();
  } else {
    // ------------------------------------------------------------------ elementwise
    const int grp = warp >> 2;            // warpgroup
    const int t = threadIdx.x & 127;      // token of the block / TMEM lane
    const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const float inv_tau_sqrt_d = 1.0f / (p.tau_s * sqrtf((float)D));
    // the retention sums: thread (c, half) for d_h = 64, thread c over all 128 tokens for 128
    const int c = D == 64 ? (t & 63) : t;
    const int half = D == 64 ? (t >> 6) : 0;
    constexpr int TPT = D == 64 ? 64 : 128;  // tokens per thread of the retention sums
    bool ok = true, my_clamp = false;
    // A block's scalars: p1_t . p2_t, |p1_t|^2, |p2_t|^2 per token, and per channel L_m and
    // (d_h = 64) the sum over the second half or (128) L_end
    auto scalars = [&](int it) {
      return reinterpret_cast<float*>(smem + C::OFF_SC + (C::AHEAD ? (it & 1) * C::SCB : 0));
    };
    // The sums of block it, once it is loaded: log2 alpha in place of alpha (0 past T; every
    // group), then Ask Self's sums (the groups but the last) beside the channels' inclusive
    // running sums L_t in place of log2 alpha (the last group; d_h = 64: the second half's
    // relative to its start).  The running sums are one chain per channel: with the logarithms
    // on the same four warps they took 3900 cycles of a block's 10600.  Visible after the
    // warpgroups' next barrier.
    auto sums = [&](int it) {
      const int t0 = (blk_first + it) * LT, st = it % C::STAGES;
      uint8_t* const sg = smem + st * C::STAGE;
      float* const al = reinterpret_cast<float*>(sg + C::OFF_A);
      float* const s_dot = scalars(it);
      float* const l_a = s_dot + 3 * LT;
      float* const l_b = l_a + LT;
      ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(B_LOAD + st), (it / C::STAGES) & 1, ab));
      if (ok) {
#pragma unroll
        for (int i0 = 0; i0 < LT * D / 4; i0 += C::EW) {
          const int i = i0 + threadIdx.x;  // 16-byte group of the tile, of token (i / 8) % 128
          const bool live = t0 + ((i >> 3) & 127) < p.T;
          float4 v = reinterpret_cast<float4*>(al)[i];
          v.x = live ? __log2f(v.x) : 0.f;
          v.y = live ? __log2f(v.y) : 0.f;
          v.z = live ? __log2f(v.z) : 0.f;
          v.w = live ? __log2f(v.w) : 0.f;
          reinterpret_cast<float4*>(al)[i] = v;
        }
      }
      ew_sync<NG>();
      if (!ok) return;
      if (grp < NG - 1) {
        ask_self_sums<D, NG == 2 ? 7 : 0>(sg + C::OFF_P1, sg + C::OFF_P2, t,
                                          NG == 2 ? 7 : 1 << grp, s_dot, s_dot + LT, s_dot + 2 * LT);
      } else {
        float lsum = 0.f;
        for (int i0 = 0; i0 < TPT; i0 += 16) {
          float la[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) la[u] = al[al_swz(half * 64 + i0 + u, c)];
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            lsum += la[u];
            al[al_swz(half * 64 + i0 + u, c)] = lsum;
          }
          if (D == 128 && i0 == 48) l_a[c] = lsum;  // L at the 64th token
        }
        if (D == 64)
          (half == 0 ? l_a : l_b)[c] = lsum;
        else
          l_b[c] = lsum;
      }
    };
    if (C::AHEAD) sums(0);
    for (int blk = blk_first; blk < blk_end; ++blk) {
      const int it = blk - blk_first;
      const uint32_t ph = it & 1;
      const int t0 = blk * LT;
      const int st = it % C::STAGES;
      uint8_t* const sg = smem + st * C::STAGE;
      uint8_t* const p1s = sg + C::OFF_P1;
      uint8_t* const p2s = sg + C::OFF_P2;
      float* const al = reinterpret_cast<float*>(sg + C::OFF_A);
      const float* const s_dot = scalars(it);
      const float* const s_n1 = s_dot + LT;
      const float* const s_n2 = s_n1 + LT;
      const float* const l_a = s_n2 + LT;
      const float* const l_b = l_a + LT;
      auto al_at = [&](int tok, int ch) -> float& {  // [D / 32][128][32] fp32, 128-byte swizzle
        return al[al_swz(tok, ch)];
      };
      if (!C::AHEAD) sums(it);
      ew_sync<NG>();
      float l_end = 0.f;  // channel t's L at the block's last token (t < D)
      if (ok) {
        if (t < D) l_end = D == 64 ? l_a[c] + l_b[c] : l_b[c];
        // Qs, KL and the state are single buffers: the last block's state product (the last
        // reader of KL; Qs's reader precedes B_E) must be done before they are written
        if (SEQ && blk > 0) {
          ok = __all_sync(0xffffffffu, mbar_wait(bar(B_STATE), (blk - 1) & 1, ab));
          tc_fence_after();
        }
      }
      if (ok) {
        // ---- the operands of token t over the group's channels, 8 per 16-byte access: Qm
        // and Km in place of p1 and p2, Qs, KL (DELTA: KL in place of p2; BOTH: and Qs of p1)
        float s1 = 0.f, s2 = 0.f;  // rows past T give zero operands
        if (t0 + t < p.T) {
          const float S = 1.0f / (1.0f + __expf(-s_dot[t] * inv_tau_sqrt_d));
          s1 = S * rsqrtf(s_n1[t]);
          s2 = S * rsqrtf(s_n2[t]);
        }
#pragma unroll
        for (int k0 = 0; k0 < D / 8 / NG; ++k0) {
          const int k = grp * (D / 8 / NG) + k0;
          const uint32_t off = (k >> 3) * LT * 128 + t * 128 + (((k & 7) ^ (t & 7)) << 4);
          uint4 a4 = make_uint4(0, 0, 0, 0);
          if (!DELTA || BOTH) a4 = *reinterpret_cast<const uint4*>(p1s + off);
          uint4 b4 = make_uint4(0, 0, 0, 0);
          b4 = *reinterpret_cast<const uint4*>(p2s + off);
          const float4 L0 = *reinterpret_cast<const float4*>(&al_at(t, 8 * k));
          const float4 L1 = *reinterpret_cast<const float4*>(&al_at(t, 8 * k + 4));
          const float4 M0 = *reinterpret_cast<const float4*>(l_a + 8 * k);
          const float4 M1 = *reinterpret_cast<const float4*>(l_a + 8 * k + 4);
          const float4 E0 = *reinterpret_cast<const float4*>(l_b + 8 * k);
          const float4 E1 = *reinterpret_cast<const float4*>(l_b + 8 * k + 4);
          const float Lv[8] = {L0.x, L0.y, L0.z, L0.w, L1.x, L1.y, L1.z, L1.w};
          const float Mv[8] = {M0.x, M0.y, M0.z, M0.w, M1.x, M1.y, M1.z, M1.w};
          const float Ev[8] = {E0.x, E0.y, E0.z, E0.w, E1.x, E1.y, E1.z, E1.w};
          const uint32_t aw[4] = {a4.x, a4.y, a4.z, a4.w}, bw[4] = {b4.x, b4.y, b4.z, b4.w};
          uint32_t qm[4], km[4], qs[4], kl[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&aw[e]));
            const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bw[e]));
            float r[2][4];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int ch = 2 * e + u;
              // the second half's sums (d_h = 64) are relative to the half's start
              const float L = Lv[ch] + ((D == 64 && t >= 64) ? Mv[ch] : 0.f);
              const float xv = u ? x.y : x.x, yv = u ? y.y : y.x;
              if (!DELTA) {
                float dm = L - Mv[ch];  // log2 of a_t / a_m
                if (fabsf(dm) > kClampLog2) {
                  dm = copysignf(kClampLog2, dm);
                  my_clamp = true;
                }
                r[u][0] = xv * s1 * ex2_approx(dm);      // Qm
                r[u][1] = yv * s2 * ex2_approx(-dm);     // Km
              }
              if (!DELTA || BOTH) r[u][2] = xv * s1 * ex2_approx(L);  // Qs (factor <= 1)
              if (MODE != MODE_OUT) {  // KL (factor <= 1)
                const float Le = D == 64 ? Mv[ch] + Ev[ch] : Ev[ch];
                r[u][3] = yv * s2 * ex2_approx(Le - L);
              }
            }
            if (!DELTA) {
              qm[e] = pack_bf16x2(r[0][0], r[1][0]);
              km[e] = pack_bf16x2(r[0][1], r[1][1]);
            }
            if (!DELTA || BOTH) qs[e] = pack_bf16x2(r[0][2], r[1][2]);
            if (MODE != MODE_OUT) kl[e] = pack_bf16x2(r[0][3], r[1][3]);
          }
          if (!DELTA) {
            *reinterpret_cast<uint4*>(p1s + off) = make_uint4(qm[0], qm[1], qm[2], qm[3]);
            *reinterpret_cast<uint4*>(p2s + off) = make_uint4(km[0], km[1], km[2], km[3]);
          }
          if (!DELTA || BOTH)
            *reinterpret_cast<uint4*>((BOTH ? p1s : smem + C::OFF_QS) + off) =
                make_uint4(qs[0], qs[1], qs[2], qs[3]);
          if (MODE != MODE_OUT)
            *reinterpret_cast<uint4*>(smem + C::OFF_KL + off) =
                make_uint4(kl[0], kl[1], kl[2], kl[3]);
        }
        fence_async_smem();
        mbar_arrive(bar(B_OPS));
      }
      if (C::IN_C0) ew_sync<NG>();  // the scalars have been read: C0 takes their place
      if (DELTA) {
        // the block's state (and adjoint) contribution and decay, to the workspace
        ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(B_STATE), 0, ab));
        tc_fence_after();
        constexpr int CG = NC / NG;  // columns per group
        const bool upper = BOTH && t >= 64;  // rows of Qs^T dY, in columns 64 .. 127
        if (ok && (t < D || BOTH)) {
          uint32_t z[32];
          const uint32_t col = trow + C::COL_C + (BOTH && (warp & 3) >= 2 ? NC : 0) + grp * CG;
          if constexpr (CG == 32)
            tmem_ld32(col, z);
          else
            tmem_ld16(col, *reinterpret_cast<uint32_t(*)[16]>(z));
          tmem_ld_wait();
          const long long row = (long long)(bhs * nb + blk) * D + (upper ? t - 64 : t);
          float* dst = (upper ? cp.dQ : cp.dC) + row * 64 + grp * CG;
#pragma unroll
          for (int k = 0; k < CG / 8; ++k) st_global_32(dst + 8 * k, z + 8 * k);
          if (grp == 0 && !upper) cp.g[row] = ex2_approx(l_end);
        }
        continue;
      }
      if (SEQ && ok) {
        // ---- the state after the last block (complete, waited above): its bf16 copy, then
        // decayed by a_L
        if (t < D) {  // (whole warps)
          uint32_t z[16];
          if (blk > 0) {
            tmem_ld16(trow + C::COL_C + grp * 16, z);
            tmem_ld_wait();
          } else {
#pragma unroll
            for (int n = 0; n < 16; ++n) z[n] = 0u;
          }
          uint8_t* crow = smem + C::OFF_C0 + t * 128;
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              w[e] = pack_bf16x2(__uint_as_float(z[8 * k + 2 * e]),
                                 __uint_as_float(z[8 * k + 2 * e + 1]));
            *reinterpret_cast<uint4*>(crow + (((2 * grp + k) ^ (t & 7)) << 4)) =
                make_uint4(w[0], w[1], w[2], w[3]);
          }
          if (blk > 0) {
            const float decay = ex2_approx(l_end);
#pragma unroll
            for (int n = 0; n < 16; ++n) z[n] = __float_as_uint(__uint_as_float(z[n]) * decay);
            tmem_st16(trow + C::COL_C + grp * 16, z);
            tmem_st_wait();
          }
        }
        fence_async_smem();
        tc_fence_before();
        mbar_arrive(bar(B_C0));
      }
      // ---- S masked to the strictly earlier tokens, packed to bf16
      ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(B_S), ph, ab));
      if (ok) {
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < LT / NG; c0 += 32) {
          const int col = grp * (LT / NG) + c0;
          uint32_t pk[16];
          if (col <= (warp & 3) * 32) {  // some column of the warp's rows is unmasked
            uint32_t s[32];
            tmem_ld32(trow + C::COL_S + col, s);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              const float lo = (col + j < t) ? __uint_as_float(s[j]) : 0.f;
              const float hi = (col + j + 1 < t) ? __uint_as_float(s[j + 1]) : 0.f;
              pk[j >> 1] = pack_bf16x2(lo, hi);
            }
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) pk[j] = 0u;
          }
          tmem_st16(trow + C::COL_P + (col >> 1), pk);
        }
        tmem_st_wait();
        tc_fence_before();
        mbar_arrive(bar(B_A));
      }
      if (C::AHEAD && blk + 1 < blk_end) sums(it + 1);
      // ---- Y = I~ + E, staged in p1's tile (stored by the TMA warp)
      ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(B_E), ph, ab));
      if (ok) {
        tc_fence_after();
        constexpr int CG = NC / NG;
        uint32_t z[CG];
        if constexpr (CG == 32)
          tmem_ld32(trow + C::COL_E + grp * CG, z);
        else
          tmem_ld16(trow + C::COL_E + grp * CG, z);
        tmem_ld_wait();
        const uint8_t* vrow = sg + C::OFF_V + t * 128;
        uint8_t* yrow = sg + C::OFF_P1 + t * 128;
#pragma unroll
        for (int k0 = 0; k0 < CG / 8; ++k0) {
          const int k = grp * (CG / 8) + k0;
          const uint4 vv = *reinterpret_cast<const uint4*>(vrow + ((k ^ (t & 7)) << 4));
          const uint32_t vw[4] = {vv.x, vv.y, vv.z, vv.w};
          uint32_t yw[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 vf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&vw[e]));
            yw[e] = pack_bf16x2(vf.x + __uint_as_float(z[8 * k0 + 2 * e]),
                                vf.y + __uint_as_float(z[8 * k0 + 2 * e + 1]));
          }
          *reinterpret_cast<uint4*>(yrow + ((k ^ (t & 7)) << 4)) =
              make_uint4(yw[0], yw[1], yw[2], yw[3]);
        }
        fence_async_smem();
        tc_fence_before();
        mbar_arrive(bar(B_EPI + st));
      }
    }
    if (my_clamp) atomicExch(clamped, 1);
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *clamped && p.dev_status && !*abort_flag)
    atomicExch(p.dev_status, (int)RELATION_ERR_UNSUPPORTED);
  if (warp == C::W_MMA) {
    tc_fence_after();
    tmem_dealloc(tmem, C::TMEM);
  }
}

// Scan of the state over the blocks of one (head, split), for the chunk-parallel forms:
// C_0(0) = 0, C_0(b + 1) = Diag(g_b) C_0(b) + dC_b; every C_0(b) is written in bf16 over the
// first half of its own row of dC_b (rows of 64 bf16 at a pitch of 256 bytes: the B operand of
// the block's products after a swizzled TMA load).  A warp owns a channel's 64 columns, two
// per lane; it has read a row (__syncwarp) before it writes it, the loads of the next P
// blocks in flight while P are combined.
//   REV (the backward): from the last block down, the state's adjoint leaving block b,
//   dC(nb - 1) = 0, dC(b - 1) = Diag(g_b) dC(b) + dQ_b (dQ_b = Qs_b^T dY_b), in place of dQ.
template <int D, bool REV>
__device__ __forceinline__ void scan_blocks(float* rows, const float* g, int nb, int bhs, int c,
                                            int n) {
  constexpr int P = 16;
  const long long base = (long long)bhs * nb * D + c;  // row of block blk: base + blk D
  auto load = [&](int b0, float2 (&dv)[P], float (&gv)[P]) {
#pragma unroll
    for (int u = 0; u < P; ++u) {
      const int blk = REV ? nb - 1 - (b0 + u) : b0 + u;
      dv[u] = make_float2(0.f, 0.f);
      gv[u] = 1.f;
      if (blk >= 0 && blk < nb) {
        const long long row = base + (long long)blk * D;
        dv[u] = *reinterpret_cast<const float2*>(rows + row * 64 + n);
        gv[u] = g[row];
      }
    }
  };
  float2 st = make_float2(0.f, 0.f), cur[P];
  float gc[P];
  load(0, cur, gc);
  for (int b0 = 0; b0 < nb; b0 += P) {
    float2 nxt[P];
    float gn[P];
    load(b0 + P, nxt, gn);
    __syncwarp();  // the warp has read rows b0 .. b0 + P - 1 (a round ago)
#pragma unroll
    for (int u = 0; u < P; ++u) {
      const int i = b0 + u;
      if (i < nb) {
        const int blk = REV ? nb - 1 - i : i;
        const long long row = base + (long long)blk * D;
        reinterpret_cast<__nv_bfloat162*>(rows + row * 64)[n >> 1] =
            __floats2bfloat162_rn(st.x, st.y);
        st = make_float2(fmaf(gc[u], st.x, cur[u].x), fmaf(gc[u], st.y, cur[u].y));
      }
    }
#pragma unroll
    for (int u = 0; u < P; ++u) {
      cur[u] = nxt[u];
      gc[u] = gn[u];
    }
  }
}

// CTAs of 8 channels; with BOTH the second half of the grid scans the adjoints.
template <int D, bool BOTH>
__global__ void __launch_bounds__(256) scan_kernel(LinCp cp, int ctas) {
  const bool rev = BOTH && (int)blockIdx.x >= ctas;
  const int w = (int)blockIdx.x - (rev ? ctas : 0);
  const int c = (w % (D / 8)) * 8 + (int)(threadIdx.x >> 5), n = (int)(threadIdx.x & 31) * 2;
  if (rev)
    scan_blocks<D, true>(cp.dQ, cp.g, cp.nb, w / (D / 8), c, n);
  else
    scan_blocks<D, false>(cp.dC, cp.g, cp.nb, w / (D / 8), c, n);
}

// Workspace of the chunk-parallel forward: dC and g per (head, split, block) (see LinCp).  The
// size also holds bf16 rows for nb + 1 states per (head, split), which the scan now keeps in
// dC's rows: the backward's second array of fp32 rows takes that place.
static size_t cp_bytes(long long heads, long long nb, int d, LinCp* out, void* base) {
  const long long rows = heads * nb * d, rows_c0 = heads * (nb + 1) * d;
  const size_t b_dc = align256((size_t)rows * 64 * 4), b_g = align256((size_t)rows * 4);
  const size_t b_c0 = align256((size_t)rows_c0 * 64 * 2);
  if (out) {
    uint8_t* q = static_cast<uint8_t*>(base);
    out->dC = reinterpret_cast<float*>(q);
    out->g = reinterpret_cast<float*>(q + b_dc);
    out->dQ = nullptr;
  }
  return b_dc + b_g + b_c0;
}

template <int D, int MODE>
static cudaError_t set_smem() {
  return cudaFuncSetAttribute(lin_tc_fwd_kernel<D, MODE>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D, MODE>::SMEM);
}

template <int D>
static cudaError_t fwd_t(const LinearProblem& lp, void* workspace, cudaStream_t s) {
  const bool cp_path = workspace != nullptr;
  cudaError_t e;
  if ((e = cp_path ? set_smem<D, MODE_DELTA>() : set_smem<D, MODE_SEQ>()) != cudaSuccess ||
      (cp_path && (e = set_smem<D, MODE_OUT>()) != cudaSuccess)) {
    note_failure("linear chunked forward: shared memory attribute");
    return e;
  }
  Problem p{};  // the bf16 tensor-map helper's view of the shapes
  p.B = lp.B; p.T = lp.T; p.H = lp.H; p.d = lp.d;
  p.sB = lp.sB; p.sT = lp.sT; p.sH = lp.sH;
  const int nb = (lp.T + LT - 1) / LT;
  const long long heads = (long long)lp.B * lp.H * (D / NC);
  LinCp cp{};
  cp.nb = nb;
  CUtensorMap m1, m2, mv, ma, my, mc;
  if (!tc::make_tmap_bf16(&m1, lp.p1, p, LT) || !tc::make_tmap_bf16(&m2, lp.p2, p, LT) ||
      !tc::make_tmap_bf16(&mv, lp.v, p, LT) || !tc::make_tmap_bf16(&my, lp.y, p, 32) ||
      !make_tmap_alpha(&ma, lp, true)) {
    note_failure("linear chunked forward: TMA descriptors");
    return cudaErrorInvalidValue;
  }
  mc = m1;  // unused by the sequential mode
  if (cp_path) {
    cp_bytes(heads, nb, D, &cp, workspace);
    if (!make_tmap_c0(&mc, cp.dC, heads * nb * D, D)) {
      note_failure("linear chunked forward: TMA descriptor of the workspace");
      return cudaErrorInvalidValue;
    }
  }
  if (!cp_path) {
    if (heads > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    using C = Cfg<D, MODE_SEQ>;
    lin_tc_fwd_kernel<D, MODE_SEQ>
        <<<(unsigned)heads, C::THREADS, C::SMEM, s>>>(m1, m2, mv, mv, ma, my, mc, lp, cp);
  } else {
    const long long grid = heads * nb, ctas = heads * (D / 8);
    if (grid > 0x7fffffffLL || ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    using CD = Cfg<D, MODE_DELTA>;
    using CO = Cfg<D, MODE_OUT>;
    lin_tc_fwd_kernel<D, MODE_DELTA>
        <<<(unsigned)grid, CD::THREADS, CD::SMEM, s>>>(m1, m2, mv, mv, ma, my, mc, lp, cp);
    if ((e = cudaGetLastError()) != cudaSuccess) { note_failure("linear chunked forward: launch"); return e; }
    scan_kernel<D, false><<<(unsigned)ctas, 256, 0, s>>>(cp, (int)ctas);
    if ((e = cudaGetLastError()) != cudaSuccess) { note_failure("linear chunked forward: launch"); return e; }
    lin_tc_fwd_kernel<D, MODE_OUT>
        <<<(unsigned)grid, CO::THREADS, CO::SMEM, s>>>(m1, m2, mv, mv, ma, my, mc, lp, cp);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) note_failure("linear chunked forward: launch");
  return e;
}

// The state passes the chunked backward needs (relation_linear_tc_bwd.cu), in the workspace
// laid out by bwd_bytes: the forward's states entering every block (bf16, in dC's rows) and the
// state's adjoint leaving every block (bf16, in dQ's rows).  Two launches: the blocks'
// contributions to both, and both scans.
size_t bwd_bytes(long long heads, long long nb, int d, LinCp* cp, void* base) {
  const size_t f = cp_bytes(heads, nb, d, cp, base);
  // dQ's fp32 rows fill what the forward's nb + 1 and the adjoints' nb bf16 rows would take
  if (cp)
    cp->dQ = reinterpret_cast<float*>(static_cast<uint8_t*>(base) +
                                      align256((size_t)(heads * nb * d) * 64 * 4) +
                                      align256((size_t)(heads * nb * d) * 4));
  return f + align256((size_t)(heads * nb * d) * 64 * 2);
}

cudaError_t launch_states(const LinearProblem& lp, const void* dy, void* workspace,
                          cudaStream_t s) {
  constexpr int D = 64;
  cudaError_t e;
  if ((e = set_smem<D, MODE_BOTH>()) != cudaSuccess) {
    note_failure("linear chunked backward: shared memory attribute");
    return e;
  }
  Problem p{};
  p.B = lp.B; p.T = lp.T; p.H = lp.H; p.d = lp.d;
  p.sB = lp.sB; p.sT = lp.sT; p.sH = lp.sH;
  const int nb = (lp.T + LT - 1) / LT;
  const long long heads = (long long)lp.B * lp.H;
  LinCp cp{};
  cp.nb = nb;
  bwd_bytes(heads, nb, D, &cp, workspace);
  CUtensorMap m1, m2, mv, mg, ma;
  if (!tc::make_tmap_bf16(&m1, lp.p1, p, LT) || !tc::make_tmap_bf16(&m2, lp.p2, p, LT) ||
      !tc::make_tmap_bf16(&mv, lp.v, p, LT) || !tc::make_tmap_bf16(&mg, dy, p, LT) ||
      !make_tmap_alpha(&ma, lp, true)) {
    note_failure("linear chunked backward: TMA descriptors");
    return cudaErrorInvalidValue;
  }
  const long long grid = heads * nb, ctas = heads * (D / 8);
  if (grid > 0x7fffffffLL || 2 * ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  // (the Y and state maps are unused in this mode; m1 stands in)
  using C = Cfg<D, MODE_BOTH>;
  lin_tc_fwd_kernel<D, MODE_BOTH>
      <<<(unsigned)grid, C::THREADS, C::SMEM, s>>>(m1, m2, mv, mg, ma, m1, m1, lp, cp);
  if ((e = cudaGetLastError()) != cudaSuccess) { note_failure("linear chunked backward: launch"); return e; }
  scan_kernel<D, true><<<(unsigned)(2 * ctas), 256, 0, s>>>(cp, (int)ctas);
  if ((e = cudaGetLastError()) != cudaSuccess) note_failure("linear chunked backward: launch");
  return e;
}

}  // namespace lintc

bool linear_tc_supports(const LinearProblem& p) {
  return p.dtype == RELATION_BF16 && (p.d == 64 || p.d == 128) && p.sB % 8 == 0 &&
         p.sT % 8 == 0 && p.sH % 8 == 0;
}

size_t linear_tc_workspace_bytes(const LinearProblem& p) {
  if (!linear_tc_supports(p)) return 0;
  const long long heads = (long long)p.B * p.H * (p.d / lintc::NC);
  const long long nb = (p.T + lintc::LT - 1) / lintc::LT;
  return lintc::cp_bytes(heads, nb, p.d, nullptr, nullptr);
}

cudaError_t launch_linear_tc_fwd(const LinearProblem& p, void* workspace, cudaStream_t s) {
  if (!linear_tc_supports(p)) return cudaErrorInvalidValue;
  return p.d == 64 ? lintc::fwd_t<64>(p, workspace, s) : lintc::fwd_t<128>(p, workspace, s);
}

}  // namespace rel
