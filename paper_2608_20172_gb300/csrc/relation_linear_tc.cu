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
// whose phases fill this one's waits.  The one-block modes' CTAs are as many as fit and take
// blocks in steps of the grid; every part of the next block's inputs is loaded as soon as its
// place is free (a CTA per block, with its launch and its loads exposed, took 1.1 to 1.2 times as
// long).  With one group (one CTA per SM) the sequential walk took 126 us at B 8, H 12, T 2048,
// d 64; four groups 93; with the logarithms on every warp, the next block's sums taken while the
// output product runs and the stores on the TMA warp 82; with one instruction per logarithm and
// no test per element for the clamp and the mask 76.  At B 1, H 12, T 32768 DELTA, the scan and
// OUT took 140, 27 and 177 us, now 57, 15 and 67 (5.1 TB/s in DELTA, half of the issue slots in
// OUT; in head order, and both from the first block on, 64 and 72).
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
  // p1, p2, alpha; and I~ (dY, the state), which the one-block modes await on their own
  static constexpr uint32_t LOAD_PA = 2 * PT + AT;
  static constexpr uint32_t LOAD_V =
      VT + (MODE == MODE_OUT ? C0T : 0) + (MODE == MODE_BOTH ? VT : 0);
  // TMEM columns: S 128 | E 64 | P 64 (S masked, bf16) | C 64; DELTA: C 64 (BOTH: 128) alone
  static constexpr int COL_S = 0, COL_E = 128, COL_P = 192, COL_C = DELTA ? 0 : 256;
  static constexpr int TMEM = SEQ ? 512 : (DELTA ? 128 : 256);
  static_assert(SCB <= C0T, "scalars in the C0 tile");
  static_assert(CTAS * (SMEM + 1024) <= 233472, "shared memory");
};

// 32 bytes to global memory (one sector); p 32-byte aligned (ws_base)
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
  // SEQ: one CTA per (head, split) over its blocks; DELTA / BOTH / OUT: any block, in steps of
  // the grid
  const int n_it =
      SEQ ? nb : (p.B * p.H * NSPLIT * nb - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
  struct Where {
    int blk, bhs, split, h, b;
  };
  auto where = [&](int it) -> Where {
    // The heads of a block of tokens side by side, as they lie in memory; OUT and BOTH from the
    // last tokens back, which DELTA, and the forward before a backward, have read last and left
    // in L2
    const int n = (int)(blockIdx.x + it * gridDim.x);
    const int item =
        MODE == MODE_OUT || BOTH ? p.B * p.H * NSPLIT * nb - 1 - n : n;
    Where w;
    if (SEQ) {
      w.bhs = (int)blockIdx.x;
      w.blk = it;
      const int bh = w.bhs / NSPLIT;
      w.split = w.bhs - bh * NSPLIT;
      w.b = bh / p.H;
      w.h = bh - w.b * p.H;
    } else {
      const int hs = p.H * NSPLIT, tb = item / hs, e = item - tb * hs;
      w.b = tb / nb;
      w.blk = tb - w.b * nb;
      w.h = e / NSPLIT;
      w.split = e - w.h * NSPLIT;
      w.bhs = (w.b * p.H + w.h) * NSPLIT + w.split;
    }
    return w;
  };

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
  pdl_wait();

  if (warp == C::W_TMA) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      // Y of block it (staged in its p1 tile; OUT: in Qs) by TMA, once every elementwise
      // thread has written its part and read the stage's I~
      auto put_y = [&](int it) {
        const int st = it % C::STAGES;
        const Where w = where(it);
        for (int q = 0; q < LT && w.blk * LT + q < p.T; q += 32)
          tma_store_4d(&tmY, sb + (SEQ ? st * C::STAGE + C::OFF_P1 : C::OFF_QS) + q * 128,
                       w.split * NC, w.blk * LT + q, w.h, w.b);
        tma_store_commit();
      };
      auto store_y = [&](int it) -> bool {
        if (!mbar_wait(bar(B_EPI + it % C::STAGES), (it / C::STAGES) & 1, ab)) return false;
        put_y(it);
        tma_store_wait_read_all();  // before the stage is loaded again (or the CTA exits)
        return true;
      };
      // the parts of block it's inputs, to stage base sg on barrier lb
      auto load_p = [&](const Where& w, uint32_t sg, uint32_t lb) {
        for (int kb = 0; kb < C::KB; ++kb) {
          tma_load_4d(sg + C::OFF_P1 + kb * LT * 128, &tmP1, lb, kb * 64, w.blk * LT, w.h, w.b);
          tma_load_4d(sg + C::OFF_P2 + kb * LT * 128, &tmP2, lb, kb * 64, w.blk * LT, w.h, w.b);
        }
      };
      auto load_a = [&](const Where& w, uint32_t sg, uint32_t lb) {
        for (int k = 0; k < D / 32; ++k)
          tma_load_4d(sg + C::OFF_A + k * LT * 128, &tmA, lb, k * 32, w.blk * LT, w.h, w.b);
      };
      auto load_v = [&](const Where& w, uint32_t sg, uint32_t lb) {
        tma_load_4d(sg + C::OFF_V, &tmV, lb, w.split * NC, w.blk * LT, w.h, w.b);
        if (BOTH) tma_load_4d(sg + C::OFF_G, &tmG, lb, w.split * NC, w.blk * LT, w.h, w.b);
        if (MODE == MODE_OUT)  // the state the block starts from, in the MN-major B layout
          tma_load_2d(sb + C::OFF_C0, &tmC0, lb, 0, (w.bhs * nb + w.blk) * D);
      };
      int issued = 0;
      bool ok = true;
      if constexpr (SEQ) {
        for (int it = 0; it < n_it; ++it) {
          const int st = it % C::STAGES, use = it / C::STAGES;
          // the stage's previous block: its MMAs are done and its output is stored
          if (use > 0 && (!(ok = store_y(it - C::STAGES)) ||
                          !(ok = mbar_wait(bar(B_FREE + st), (use - 1) & 1, ab))))
            break;
          const Where w = where(it);
          const uint32_t sg = sb + st * C::STAGE, lb = bar(B_LOAD + st);
          mbar_arrive_expect_tx(lb, C::LOAD_PA + C::LOAD_V);
          load_p(w, sg, lb);
          load_a(w, sg, lb);
          load_v(w, sg, lb);
          issued = it + 1;
        }
        for (int it = max(0, n_it - C::STAGES); ok && it < n_it; ++it) ok = store_y(it);
        if (ab.raised())  // copies in flight land before the CTA releases its shared memory
          for (int it = issued - C::STAGES > 0 ? issued - C::STAGES : 0; it < issued; ++it)
            drain_wait(bar(B_LOAD + it % C::STAGES), (it / C::STAGES) & 1);
      } else {
        // One stage, whose parts are loaded for the next block as this one lets go of them:
        // alpha when the operands are made, p1 and p2 when their product is done (DELTA, BOTH:
        // with I~ and dY, when the state product is), I~ and the state after the epilogue
        const uint32_t lb = bar(B_LOAD), lv = bar(B_LOADV);
        mbar_arrive_expect_tx(lb, C::LOAD_PA);
        load_p(where(0), sb, lb);
        load_a(where(0), sb, lb);
        mbar_arrive_expect_tx(lv, C::LOAD_V);
        load_v(where(0), sb, lv);
        issued = 1;
        for (int it = 0; ok && it < n_it; ++it) {
          const bool more = it + 1 < n_it;
          const Where nx = where(more ? it + 1 : it);
          const uint32_t ph = it & 1;
          if (more) {
            if (!(ok = mbar_wait(bar(B_OPS), ph, ab))) break;
            mbar_arrive_expect_tx(lb, C::LOAD_PA);
            load_a(nx, sb, lb);
            issued = it + 2;
            if (!(ok = mbar_wait(bar(DELTA ? B_STATE : B_S), ph, ab))) break;
            load_p(nx, sb, lb);
            if (DELTA) {
              mbar_arrive_expect_tx(lv, C::LOAD_V);
              load_v(nx, sb, lv);
            }
          }
          if (!DELTA) {
            if (!(ok = mbar_wait(bar(B_EPI), ph, ab))) break;
            put_y(it);
            if (more) {
              mbar_arrive_expect_tx(lv, C::LOAD_V);
              load_v(nx, sb, lv);
            }
            tma_store_wait_read_all();
            mbar_arrive(bar(B_QFREE));  // Qs may be written again
          }
        }
        if (ab.raised()) {  // copies in flight land before the CTA exits
          drain_wait(bar(B_LOAD), (issued - 1) & 1);
          drain_wait(bar(B_LOADV), (issued - 1) & 1);
        }
      }
    }
  } else if (warp == C::W_MMA) {
    // ------------------------------------------------------------------ MMA issuer
    constexpr uint32_t id_s = idesc_bf16_f32(128, 128, false, false);
    constexpr uint32_t id_e = idesc_bf16_f32(128, NC, false, true);
    constexpr uint32_t id_c = idesc_bf16_f32(128, BOTH ? 2 * NC : NC, true, true);
    bool ok = true;
    for (int it = 0; ok && it < n_it; ++it) {
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
        if (!(ok = mbar_wait_warp(bar(SEQ ? B_C0 : B_LOADV), ph, ab))) break;
        tc_fence_after();
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
      if (DELTA && !(ok = mbar_wait_warp(bar(B_LOADV), ph, ab))) break;
      if (MODE != MODE_OUT) {
        // SEQ: C += KL^T I~ (C decayed by the threads); DELTA: the block's own sum; BOTH:
        // [KL | Qs]^T [I~ | dY], whose diagonal quarters are the two contributions
#pragma unroll
        for (int kk = 0; kk < LT / 16; ++kk)
          mma_ss_w(tmem + C::COL_C,
                   smem_desc_sw128(sb + C::OFF_KL + kk * 16 * 128, LT * 128, 1024),
                   smem_desc_sw128(sg + C::OFF_V + kk * 16 * 128, LT * 128, 1024), id_c,
                   ((SEQ && it > 0) || kk > 0) ? 1u : 0u);
        mma_commit_w(bar(B_STATE));
      }
      if (SEQ) mma_commit_w(bar(B_FREE + st));
    }
    // SEQ: the last commits land before the CTA exits (EW warps have waited for the others)
    if (SEQ && ok)
      for (int it = max(0, n_it - C::STAGES); it < n_it; ++it)
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
      const int t0 = where(it).blk * LT, st = it % C::STAGES;
      uint8_t* const sg = smem + st * C::STAGE;
      float* const al = reinterpret_cast<float*>(sg + C::OFF_A);
      float* const s_dot = scalars(it);
      float* const l_a = s_dot + 3 * LT;
      float* const l_b = l_a + LT;
      ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(B_LOAD + st), (it / C::STAGES) & 1, ab));
      auto logs = [&](bool full) {
#pragma unroll
        for (int i0 = 0; i0 < LT * D / 4; i0 += C::EW) {
          const int i = i0 + threadIdx.x;  // 16-byte group of the tile, of token (i / 8) % 128
          const bool live = full || t0 + ((i >> 3) & 127) < p.T;
          float4 v = reinterpret_cast<float4*>(al)[i];
          v.x = live ? log2_alpha(v.x) : 0.f;
          v.y = live ? log2_alpha(v.y) : 0.f;
          v.z = live ? log2_alpha(v.z) : 0.f;
          v.w = live ? log2_alpha(v.w) : 0.f;
          reinterpret_cast<float4*>(al)[i] = v;
        }
      };
      if (ok) {
        if (t0 + LT <= p.T)
          logs(true);
        else
          logs(false);
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
    for (int it = 0; it < n_it; ++it) {
      const uint32_t ph = it & 1;
      const Where w = where(it);
      const int t0 = w.blk * LT;
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
        if (SEQ && it > 0) {
          ok = __all_sync(0xffffffffu, mbar_wait(bar(B_STATE), (it - 1) & 1, ab));
          tc_fence_after();
        }
        if (MODE == MODE_OUT && it > 0)  // Qs: the last block's Y has left it
          ok = __all_sync(0xffffffffu, mbar_wait(bar(B_QFREE), (it - 1) & 1, ab));
      }
      if (ok) {
        // ---- the operands of token t over the group's channels, 8 per 16-byte access: Qm
        // and Km in place of p1 and p2, Qs, KL (DELTA: KL in place of p2; BOTH: and Qs of p1)
        const float later = D == 64 && t >= 64 ? 1.f : 0.f;
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
          // L_t (the second half's sums (d_h = 64) are relative to the half's start) and log2 of
          // a_t / a_m
          float Lt[8], dm[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            Lt[i] = D == 64 ? fmaf(Mv[i], later, Lv[i]) : Lv[i];
            dm[i] = Lt[i] - Mv[i];
          }
          if (!DELTA) clamp_exponents(dm, my_clamp);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&aw[e]));
            const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bw[e]));
            float r[2][4];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int ch = 2 * e + u;
              const float L = Lt[ch];
              const float xv = u ? x.y : x.x, yv = u ? y.y : y.x;
              if (!DELTA) {
                r[u][0] = xv * s1 * ex2_approx(dm[ch]);   // Qm
                r[u][1] = yv * s2 * ex2_approx(-dm[ch]);  // Km
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
        ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(B_STATE), ph, ab));
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
          const long long row = (long long)(w.bhs * nb + w.blk) * D + (upper ? t - 64 : t);
          float* dst = (upper ? cp.dQ : cp.dC) + row * 64 + grp * CG;
#pragma unroll
          for (int k = 0; k < CG / 8; ++k) st_global_32(dst + 8 * k, z + 8 * k);
          if (grp == 0 && !upper) cp.g[row] = ex2_approx(l_end);
        }
        tc_fence_before();  // the sums have been read: the next block's product may start
        continue;
      }
      if (SEQ && ok) {
        // ---- the state after the last block (complete, waited above): its bf16 copy, then
        // decayed by a_L
        if (t < D) {  // (whole warps)
          uint32_t z[16];
          if (it > 0) {
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
          if (it > 0) {
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
            if (col == (warp & 3) * 32) {  // the warp's diagonal square
#pragma unroll
              for (int j = 0; j < 32; ++j) s[j] = col + j < t ? s[j] : 0u;
            }
#pragma unroll
            for (int j = 0; j < 32; j += 2)
              pk[j >> 1] = pack_bf16x2(__uint_as_float(s[j]), __uint_as_float(s[j + 1]));
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
      if (C::AHEAD && it + 1 < n_it) sums(it + 1);
      // ---- Y = I~ + E, staged in p1's tile (OUT: in Qs; stored by the TMA warp)
      ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(B_E), ph, ab));
      if (!SEQ) ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(B_LOADV), ph, ab));
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
        uint8_t* yrow = (SEQ ? sg + C::OFF_P1 : smem + C::OFF_QS) + t * 128;
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
  pdl_wait_and_launch();
  const bool rev = BOTH && (int)blockIdx.x >= ctas;
  const int w = (int)blockIdx.x - (rev ? ctas : 0);
  const int c = (w % (D / 8)) * 8 + (int)(threadIdx.x >> 5), n = (int)(threadIdx.x & 31) * 2;
  if (rev)
    scan_blocks<D, true>(cp.dQ, cp.g, cp.nb, w / (D / 8), c, n);
  else
    scan_blocks<D, false>(cp.dC, cp.g, cp.nb, w / (D / 8), c, n);
}

// Where the arrays start in a workspace, which is 16-byte aligned only: the stores of whole sectors
// (st_global_32) take 32 bytes, and rows of 256 bytes should not straddle more cache lines than
// they fill.  The up to 240 bytes this skips are in the size already: of the bf16 rows that it
// counts for nb + 1 states per (head, split), the forward uses none and the backward leaves at
// least d rows of 128 bytes.
static uint8_t* ws_base(void* base) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(base) + 255) & ~(uintptr_t)255);
}

// Workspace of the chunk-parallel forward: dC and g per (head, split, block) (see LinCp).  The
// size also holds bf16 rows for nb + 1 states per (head, split), which the scan now keeps in
// dC's rows: the backward's second array of fp32 rows takes that place.
static size_t cp_bytes(long long heads, long long nb, int d, LinCp* out, void* base) {
  const long long rows = heads * nb * d, rows_c0 = heads * (nb + 1) * d;
  const size_t b_dc = align256((size_t)rows * 64 * 4), b_g = align256((size_t)rows * 4);
  const size_t b_c0 = align256((size_t)rows_c0 * 64 * 2);
  if (out) {
    uint8_t* q = ws_base(base);
    out->dC = reinterpret_cast<float*>(q);
    out->g = reinterpret_cast<float*>(q + b_dc);
    out->dQ = nullptr;
  }
  return b_dc + b_g + b_c0;
}

// CTAs of the one-block modes: as many as are resident at once, which share the blocks evenly
static cudaError_t block_grid(long long blocks, int per_sm, unsigned* grid) {
  int dev = 0, nsm = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) {
    note_failure("linear chunked: device attributes");
    return e;
  }
  *grid = (unsigned)(blocks < (long long)per_sm * nsm ? blocks : (long long)per_sm * nsm);
  return cudaSuccess;
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
    e = launch_pdl(lin_tc_fwd_kernel<D, MODE_SEQ>, dim3((unsigned)heads), C::THREADS, C::SMEM, s, 1,
                   m1, m2, mv, mv, ma, my, mc, lp, cp);
  } else {
    using CD = Cfg<D, MODE_DELTA>;
    using CO = Cfg<D, MODE_OUT>;
    const long long ctas = heads * (D / 8);
    if (heads * nb > 0x7fffffffLL || ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    unsigned grid = 0;
    if ((e = block_grid(heads * nb, CD::CTAS, &grid)) != cudaSuccess) return e;
    static_assert(CD::CTAS == CO::CTAS, "one grid for both");
    if ((e = launch_pdl(lin_tc_fwd_kernel<D, MODE_DELTA>, dim3(grid), CD::THREADS, CD::SMEM, s, 1, m1,
                        m2, mv, mv, ma, my, mc, lp, cp)) == cudaSuccess &&
        (e = launch_pdl(scan_kernel<D, false>, dim3((unsigned)ctas), 256, 0, s, 1, cp, (int)ctas)) ==
            cudaSuccess)
      e = launch_pdl(lin_tc_fwd_kernel<D, MODE_OUT>, dim3(grid), CO::THREADS, CO::SMEM, s, 1, m1, m2,
                     mv, mv, ma, my, mc, lp, cp);
  }
  if (e != cudaSuccess) note_failure("linear chunked forward: launch");
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
    cp->dQ = reinterpret_cast<float*>(ws_base(base) + align256((size_t)(heads * nb * d) * 64 * 4) +
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
  // (the Y and state maps are unused in this mode; m1 stands in)
  using C = Cfg<D, MODE_BOTH>;
  const long long ctas = heads * (D / 8);
  if (heads * nb > 0x7fffffffLL || 2 * ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  unsigned grid = 0;
  if ((e = block_grid(heads * nb, C::CTAS, &grid)) != cudaSuccess) return e;
  if ((e = launch_pdl(lin_tc_fwd_kernel<D, MODE_BOTH>, dim3(grid), C::THREADS, C::SMEM, s, 1, m1, m2,
                      mv, mg, ma, m1, m1, lp, cp)) == cudaSuccess)
    e = launch_pdl(scan_kernel<D, true>, dim3((unsigned)(2 * ctas)), 256, 0, s, 1, cp, (int)ctas);
  if (e != cudaSuccess) note_failure("linear chunked backward: launch");
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
