// relation_simt.cu -- CUDA-core (SIMT) FlashRelation kernels, fp32 and bf16 I/O.
//
// These kernels run the exact causal Relation operator with fp32 arithmetic on the
// CUDA cores.  They serve the fp32 workloads (expf and logf, not the fast forms; the row
// statistics and the sums that cancel in two floats) and every (dtype, d_h) the tensor-core
// kernels do not cover.
//
// Work split.  A CTA of W warps owns 8 W rows of one head (queries in the forward and dQ,
// keys in dK / dV), eight per warp, and walks the other side in staged tiles of 64 rows.
// Within a warp, lane = 16 ty + tx: the products over d (U, dP) give each lane a 4 x 4 tile
// (rows 4 ty .., the tile's rows 16 i + tx), the products over the tile (z, dV, dK, dQ) a
// tile of 4 rows x D / 16 columns, so that eight 16-byte shared-memory reads feed 64
// multiply-adds (32 packed ones in the products over d).  The rows of a warp meet no other
// warp's: the weights pass between the two kinds of product through a warp-private
// [8][64] buffer.  Bound: shared-memory bandwidth and the FP32 pipe (backward: 78 % of the
// wavefronts, 58 % of the pipe), 2 + 7 products of d_h over the causal pairs (forward +
// backward); in small grids, the chain of tiles of the longest rows, which two groups of warps
// then share (two_groups, by measured lines).  Measured, B 2, H 8, T 1000, d 64, forward + backward: 1478 -> 293 us
// (forward 567 -> 80, backward tiles 920 -> 210) against a thread per quarter row (one 16-byte
// shared read per four multiply-adds, two shuffles per entry); B 1, H 2, T 128, d 32: 49 -> 9 and
// 77 -> 11 us.
//
// Forward (Sec. 5.1, App. A.3): per tile the row's Exchange entries E_ij = SiLU(U_ij) (j < i)
// update the running (m, l, z) state; the diagonal entry gives S_i = sigmoid(U_ii / tau_S)
// and is kept out of the scan.  The epilogue applies the count correction and the
// Self-Exchange split:
//   A_i = m + log l - lambda log i, g_i = sigmoid(A_i - S_i),
//   Y_i = (1 - g_i) v_i + g_i z / l,  logZ_i = logaddexp(S_i, A_i)   (App. A.3.5).
// logZ's error is a relative error of all weights of its row in the backward, so A_i is a sum
// of two floats: logZ to 2.5e-8 of 64 bits instead of 1.1e-7 (T 1000, d 64; rms over the rows),
// dL/dlambda to 1.1e-6 instead of 4.9e-6 (rms over inputs), for 1 % of the time.
//
// Backward (App. A.1.7): the Self part and D_i come from the shared row kernel
// (aux_kernels.cu); one launch holds key-stationary CTAs that accumulate dK, dV over query
// tiles and query-stationary CTAs that accumulate dQ over key tiles (together, so that a
// short sequence fills more of the GPU), both recomputing
//   P_ij = exp(E_ij - lambda log i - logZ_i), dR_ij = P_ij (dO_i . v_j - D_i),
//   dS_ij = dR_ij SiLU'(u_ij)  for j < i.
// No atomics: every output element is written by exactly one thread.
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace rel {
namespace simt {

constexpr int kTile = 64;       // rows per staged tile
constexpr int kWarpRows = 8;    // rows per warp
constexpr int PW = kTile + 4;   // row stride of the warp-private weight buffer
// shared-memory row stride of a staged tile: 16 consecutive rows' 16-byte reads spread over
// the banks (two wavefronts for 256 bytes)
template <int D>
struct Ld {
  static constexpr int V = D + 4;
};

template <typename TI>
struct IO;
template <>
struct IO<float> {
  static __device__ __forceinline__ float4 load4(const float* p) {
    return *reinterpret_cast<const float4*>(p);
  }
  static __device__ __forceinline__ float2 load2(const float* p) {
    return *reinterpret_cast<const float2*>(p);
  }
  static __device__ __forceinline__ void store4(float* p, float4 v) {
    *reinterpret_cast<float4*>(p) = v;
  }
  static __device__ __forceinline__ void store2(float* p, float2 v) {
    *reinterpret_cast<float2*>(p) = v;
  }
};
template <>
struct IO<__nv_bfloat16> {
  static __device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
    uint2 raw = *reinterpret_cast<const uint2*>(p);
    __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162*>(&raw.x);
    __nv_bfloat162 b = *reinterpret_cast<__nv_bfloat162*>(&raw.y);
    float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
    return make_float4(fa.x, fa.y, fb.x, fb.y);
  }
  static __device__ __forceinline__ float2 load2(const __nv_bfloat16* p) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
  }
  static __device__ __forceinline__ void store4(__nv_bfloat16* p, float4 v) {
    __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y);
    __nv_bfloat162 b = __floats2bfloat162_rn(v.z, v.w);
    uint2 raw;
    raw.x = *reinterpret_cast<uint32_t*>(&a);
    raw.y = *reinterpret_cast<uint32_t*>(&b);
    *reinterpret_cast<uint2*>(p) = raw;
  }
  static __device__ __forceinline__ void store2(__nv_bfloat16* p, float2 v) {
    *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(v.x, v.y);
  }
};

// The denominator is at least 1: __fdividef (2 ulp, 0 for a denominator above 2^126) takes no
// branch, so that a lane's 16 entries overlap; the IEEE division's range check kept them apart and
// costs 12 % of the forward and 5 % of the backward.  Against 64 bits over 42 inputs (d 32 to 128,
// T 33 to 2048) the outputs' errors are those with the IEEE division: Y 2.379e-7 and 2.377e-7 (rms of
// the relative errors), logZ 4.42e-8 and 4.44e-8, dQ 3.400e-7 and 3.399e-7, dK 5.087e-7 and 5.082e-7,
// dV 3.163e-7 and 3.162e-7; the rounding of the products over d and of expf decides them.
__device__ __forceinline__ float sigmoidf_acc(float x) { return __fdividef(1.0f, 1.0f + expf(-x)); }

// A lane's columns of a row of D: D = 32: 2 tx .., D = 64: 4 tx .., D = 128: 4 tx .. and
// 64 + 4 tx ..
template <int D>
struct Cols {
  static constexpr int N = D / 16;
  static constexpr int V = N < 4 ? N : 4;  // per access
  static __device__ __forceinline__ int at(int tx, int c) { return (c / V) * 64 + tx * V; }
};
template <typename TI, int D>
__device__ __forceinline__ void load_cols(const TI* row, int tx, float (&x)[D / 16]) {
  using C = Cols<D>;
#pragma unroll
  for (int c = 0; c < C::N; c += C::V) {
    if constexpr (C::V == 2) {
      const float2 t = IO<TI>::load2(row + C::at(tx, c));
      x[c] = t.x; x[c + 1] = t.y;
    } else {
      const float4 t = IO<TI>::load4(row + C::at(tx, c));
      x[c] = t.x; x[c + 1] = t.y; x[c + 2] = t.z; x[c + 3] = t.w;
    }
  }
}
template <typename TI, int D>
__device__ __forceinline__ void store_cols(TI* row, int tx, const float (&x)[D / 16]) {
  using C = Cols<D>;
#pragma unroll
  for (int c = 0; c < C::N; c += C::V) {
    if constexpr (C::V == 2)
      IO<TI>::store2(row + C::at(tx, c), make_float2(x[c], x[c + 1]));
    else
      IO<TI>::store4(row + C::at(tx, c), make_float4(x[c], x[c + 1], x[c + 2], x[c + 3]));
  }
}

// NG groups of W warps share the tiles of a CTA's rows (group g the tiles g, g + NG, ...) and add
// up their sums at the end: the NT threads of group g meet.
template <int NT, int NG>
__device__ __forceinline__ void group_sync(int g) {
  if (NG == 1)
    __syncthreads();
  else if (g == 0)
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
  else
    asm volatile("bar.sync 2, %0;" ::"n"(NT) : "memory");
}

// Stage `rows` rows from r0 of one head into shared memory as fp32 (rows >= T are zero).
// fp32 rows go by cp.async (16 bytes, zero-filled past T) and are complete after
// stage_wait and a barrier; bf16 rows are converted on the way.
template <typename TI, int D, int NT>
__device__ __forceinline__ void stage(float* dst, const TI* src, long long sT, int r0, int rows,
                                      int T, int tid) {  // tid: of the NT threads that stage it
  constexpr int LD = Ld<D>::V;
  for (int idx = tid; idx < rows * (D / 4); idx += NT) {
    const int rr = idx / (D / 4), c4 = idx % (D / 4);
    const int r = r0 + rr;
    float* to = dst + rr * LD + 4 * c4;
    if constexpr (sizeof(TI) == 4) {
      const TI* from = src + (long long)min(r, T - 1) * sT + 4 * c4;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(to)), "l"(from),
                   "r"(r < T ? 16 : 0)
                   : "memory");
    } else {
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < T) t = IO<TI>::load4(src + (long long)r * sT + 4 * c4);
      *reinterpret_cast<float4*>(to) = t;
    }
  }
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void stage_wait() {  // all but the last N groups have landed
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// s[r][i] = a_(4 ty + r) . b_(16 i + tx): rows of a (the warp's eight) and of a staged tile
template <int D>
__device__ __forceinline__ void dots(const float* a, const float* b, int ty, int tx,
                                     float (&s)[4][4]) {
  constexpr int LD = Ld<D>::V;
  float2 acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[r][i] = make_float2(0.f, 0.f);
  const float* ar = a + 4 * ty * LD;
  const float* br = b + tx * LD;
#pragma unroll 4
  for (int d = 0; d < D; d += 4) {
    float4 x[4], y[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) x[r] = *reinterpret_cast<const float4*>(ar + r * LD + d);
#pragma unroll
    for (int i = 0; i < 4; ++i) y[i] = *reinterpret_cast<const float4*>(br + 16 * i * LD + d);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        acc[r][i] = __ffma2_rn(make_float2(x[r].x, x[r].y), make_float2(y[i].x, y[i].y), acc[r][i]);
        acc[r][i] = __ffma2_rn(make_float2(x[r].z, x[r].w), make_float2(y[i].z, y[i].w), acc[r][i]);
      }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) s[r][i] = acc[r][i].x + acc[r][i].y;
}

// z[r] += sum_(k in [k0, k1)) w[4 ty + r][k] b_k over the lane's columns; k0, k1 multiples of
// 4.  MASK: only the entries with use(r, k), so that a masked row of b (which may hold
// anything) never enters, not even times zero.
template <int D, bool MASK, typename F>
__device__ __forceinline__ void axpys(const float* w, const float* b, int ty, int tx, int k0,
                                      int k1, float (&z)[4][D / 16], F use) {
  constexpr int LD = Ld<D>::V;
  const float* wr = w + 4 * ty * PW;
#pragma unroll 2
  for (int k = k0; k < k1; k += 4) {
    float4 p4[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) p4[r] = *reinterpret_cast<const float4*>(wr + r * PW + k);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float v[D / 16];
      load_cols<float, D>(b + (k + e) * LD, tx, v);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float pv = e == 0 ? p4[r].x : e == 1 ? p4[r].y : e == 2 ? p4[r].z : p4[r].w;
        if (!MASK || use(r, k + e)) {
#pragma unroll
          for (int c = 0; c < D / 16; ++c) z[r][c] = fmaf(pv, v[c], z[r][c]);
        }
      }
    }
  }
}

// Maximum that keeps a NaN (fmaxf drops it): a NaN score makes its row's scale NaN, and so all of
// the row's weights, also where no other score has been seen
__device__ __forceinline__ float max_nan(float a, float b) {
  float y;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
  return y;
}
// Sum / maximum over the 16 lanes that share a row
__device__ __forceinline__ float row_sum(float x) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __forceinline__ float row_max(float x) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) x = max_nan(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

// ---------------------------------------------------------------------------
// Forward
// ---------------------------------------------------------------------------
template <int D, int W, int NG>
constexpr size_t fwd_smem() {
  return (size_t)(kWarpRows * W + NG * 2 * kTile) * Ld<D>::V * 4 +
         (size_t)NG * W * kWarpRows * PW * 4;
}

template <typename TI, int D, int W, int NG>
__global__ void __launch_bounds__(32 * W * NG, NG == 2 && D < 128 ? 2 : 0) fwd_kernel(Problem p, int n_t) {
  constexpr int LD = Ld<D>::V, ROWS = kWarpRows * W, NT = 32 * W;
  extern __shared__ float4 smem_f4[];
  float* Qs = reinterpret_cast<float*>(smem_f4);
  const int grp = NG == 1 ? 0 : threadIdx.x / NT, tid = NG == 1 ? threadIdx.x : threadIdx.x % NT;
  float* Ks = Qs + ROWS * LD + grp * 2 * kTile * LD;
  float* Vs = Ks + kTile * LD;
  const int warp = tid >> 5, lane = tid & 31, ty = lane >> 4, tx = lane & 15;
  float* Pw = Qs + (ROWS + NG * 2 * kTile) * LD + (threadIdx.x >> 5) * kWarpRows * PW;
  const float* Qw = Qs + warp * kWarpRows * LD;
  pdl_wait();
  const int BH = p.B * p.H;
  const int qt = n_t - 1 - (int)(blockIdx.x / BH);  // most key tiles first
  const int bh = (int)(blockIdx.x % BH), b = bh / p.H, h = bh % p.H;
  const int q0 = qt * ROWS;
  const int r0 = q0 + warp * kWarpRows + 4 * ty;  // the lane's rows r0 .. r0 + 3
  const long long base = (long long)b * p.sB + (long long)h * p.sH;
  const TI* Q = reinterpret_cast<const TI*>(p.q) + base;
  const TI* K = reinterpret_cast<const TI*>(p.k) + base;
  const TI* V = reinterpret_cast<const TI*>(p.v) + base;

  float z[4][D / 16], m[4], l[4], u_self[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    m[r] = -INFINITY;
    l[r] = u_self[r] = 0.f;
#pragma unroll
    for (int c = 0; c < D / 16; ++c) z[r][c] = 0.f;
  }
  const int kend = min(p.T, q0 + ROWS);
  constexpr int STEP = NG * kTile;
  stage<TI, D, NT * NG>(Qs, Q, p.sT, q0, ROWS, p.T, threadIdx.x);
  stage_commit();
  if (grp * kTile < kend) stage<TI, D, NT>(Ks, K, p.sT, grp * kTile, kTile, p.T, tid);
  stage_commit();
  if (grp * kTile < kend) stage<TI, D, NT>(Vs, V, p.sT, grp * kTile, kTile, p.T, tid);
  stage_commit();
  stage_wait<2>();
  __syncthreads();  // Q is in
  for (int k0 = grp * kTile; k0 < kend; k0 += STEP) {
    stage_wait<1>();
    group_sync<NT, NG>(grp);  // K is in
    const int hist = q0 + warp * kWarpRows + kWarpRows - 1 - k0;  // the warp's last history key + 1
    float sc[4];
    {
      float e[4][4];
      dots<D>(Qw, Ks, ty, tx, e);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float mt = -INFINITY;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int j = k0 + 16 * i + tx;
          const float u = e[r][i] * p.inv_sqrt_d;
          const float ev = u * sigmoidf_acc(u);        // E_ij = SiLU(U_ij)
          e[r][i] = j < r0 + r ? ev : -INFINITY;
          u_self[r] = j == r0 + r ? u : u_self[r];
          mt = max_nan(mt, e[r][i]);
        }
        const float mn = max_nan(m[r], row_max(mt));
        // no history seen yet (mn = -inf): every weight is 0
        sc[r] = mn == -INFINITY ? 1.f : expf(m[r] - mn);
        float ls = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float w = mn == -INFINITY ? 0.f : expf(e[r][i] - mn);
          ls += w;
          Pw[(4 * ty + r) * PW + 16 * i + tx] = w;
        }
        l[r] = fmaf(l[r], sc[r], ls);  // this lane's share of the row sum
        m[r] = mn;
      }
    }
    group_sync<NT, NG>(grp);  // K has been read
    if (k0 + STEP < kend) stage<TI, D, NT>(Ks, K, p.sT, k0 + STEP, kTile, p.T, tid);
    stage_commit();
    stage_wait<1>();
    group_sync<NT, NG>(grp);  // V is in
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < D / 16; ++c) z[r][c] *= sc[r];
    // keys every row of the warp has in its history, then the (at most 8) mixed ones
    const int full = max(0, min(kTile, (hist - kWarpRows + 1) & ~3));
    const int some = max(0, min(kTile, (hist + 3) & ~3));
    axpys<D, false>(Pw, Vs, ty, tx, 0, full, z, [](int, int) { return true; });
    axpys<D, true>(Pw, Vs, ty, tx, full, some, z, [&](int r, int k) { return k0 + k < r0 + r; });
    group_sync<NT, NG>(grp);  // V has been read
    if (k0 + STEP < kend) stage<TI, D, NT>(Vs, V, p.sT, k0 + STEP, kTile, p.T, tid);
    stage_commit();
  }

#pragma unroll
  for (int r = 0; r < 4; ++r) {
    l[r] = row_sum(l[r]);
    u_self[r] = row_sum(u_self[r]);  // held by the lane whose key it was, 0 elsewhere
  }
  if constexpr (NG == 2) {
    // the second group's (m, l, U_ii, z) through its own tiles to the first, which finishes the rows
    float* const zs = Qs + (ROWS + 2 * kTile) * LD + (warp * kWarpRows + 4 * ty) * LD;
    float* const st = Qs + (ROWS + 3 * kTile) * LD + (warp * kWarpRows + 4 * ty) * 4;
    if (grp == 1) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        store_cols<float, D>(zs + r * LD, tx, z[r]);
        if (tx == 0) *reinterpret_cast<float4*>(st + 4 * r) = make_float4(m[r], l[r], u_self[r], 0.f);
      }
    }
    __syncthreads();
    if (grp == 1) return;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 o = *reinterpret_cast<const float4*>(st + 4 * r);
      u_self[r] += o.z;
      if (o.x == -INFINITY) continue;  // no history there
      const float mn = max_nan(m[r], o.x), a = m[r] == -INFINITY ? 0.f : expf(m[r] - mn), b2 = expf(o.x - mn);
      float zo[D / 16];
      load_cols<float, D>(zs + r * LD, tx, zo);
      m[r] = mn;
      l[r] = fmaf(l[r], a, o.y * b2);
#pragma unroll
      for (int c = 0; c < D / 16; ++c) z[r][c] = fmaf(z[r][c], a, zo[c] * b2);
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = r0 + r;
    if (row >= p.T) continue;
    const float lr = l[r], S = 1.0f / (1.0f + expf(-u_self[r] / p.tau_s));
    float g = 0.f, lz = S;
    float inv_l = 0.f, fself = 1.0f;  // F_ii = 1 - g: the Self flow
    if (row > 0 && lr > 0.f) {
      // A = m + log l - lambda log i as a sum of two floats (where it is finite): logZ's error is
      // a relative error of the whole row's weights in the backward
      Sum2 a;
      a.add(m[r]);
      a.add_log(lr, 1.f);
      a.add_log((float)(row + 1), -p.lambda);
      const float A = a.s, Alo = fabsf(A) < INFINITY ? a.c : 0.f;
      const float t = (A - S) + Alo;  // A - S
      g = 1.0f / (1.0f + expf(-t));
      fself = 1.0f / (1.0f + expf(t));
      const float x = log1pf(expf(-fabsf(t)));
      lz = t > 0.f ? A + (Alo + x) : S + x;
      inv_l = 1.0f / lr;
    }
    float y[D / 16];
    load_cols<TI, D>(V + (long long)row * p.sT, tx, y);
#pragma unroll
    for (int c = 0; c < D / 16; ++c) y[c] = (1.f - g) * y[c] + g * (z[r][c] * inv_l);
    store_cols<TI, D>(reinterpret_cast<TI*>(p.out) + base + (long long)row * p.sT, tx, y);
    if (tx == 0) {
      p.logz[(long long)bh * p.T + row] = lz;
      if (p.fself) p.fself[(long long)bh * p.T + row] = fself;
    }
  }
}

// ---------------------------------------------------------------------------
// Backward
// ---------------------------------------------------------------------------
template <int D, int W, int NG>
constexpr size_t bwd_smem() {
  return (size_t)(2 * kWarpRows * W + NG * 2 * kTile) * Ld<D>::V * 4 +
         (size_t)NG * (W * kWarpRows * PW * 4 + 3 * kTile * 4 + W * 4);
}

// P_ij and dS_ij of one Exchange pair: ci = -lambda log i - logZ_i
__device__ __forceinline__ void pair_grad(float u, float dP, float ci, float Di, float& P,
                                          float& dR, float& dS) {
  const float sg = sigmoidf_acc(u);
  const float E = u * sg;
  P = expf(E + ci);
  dR = P * (dP - Di);
  dS = dR * (sg + E * (1.f - sg));  // SiLU'(u) = sigma + E (1 - sigma)
}

// dK, dV (key-stationary): the CTA's ROWS keys over the query tiles from its first key on
template <typename TI, int D, int W, int NG>
__device__ __forceinline__ void bwd_dkdv(const Problem& p, const BwdWorkspace& ws, float* dlam_part,
                                         float* smem, int kt, int bh) {
  constexpr int LD = Ld<D>::V, ROWS = kWarpRows * W, NT = 32 * W;
  float* Ks = smem;
  float* Vs = Ks + ROWS * LD;
  const int grp = NG == 1 ? 0 : threadIdx.x / NT, tid = NG == 1 ? threadIdx.x : threadIdx.x % NT;
  float* Qs = Vs + ROWS * LD + grp * 2 * kTile * LD;
  float* Gs = Qs + kTile * LD;  // dO tile
  const int warp = tid >> 5, lane = tid & 31, ty = lane >> 4, tx = lane & 15;
  float* const after = Vs + (ROWS + NG * 2 * kTile) * LD;
  float* Pw = after + (threadIdx.x >> 5) * kWarpRows * PW;
  float* cs = after + NG * W * kWarpRows * PW + grp * 3 * kTile;  // -lambda log i - logZ_i
  float* Ds = cs + kTile;                            // D_i
  float* wl = Ds + kTile;                            // log i * F_ii (Exchange weight of dlambda)
  float* red = after + NG * (W * kWarpRows * PW + 3 * kTile);
  const int b = bh / p.H, h = bh % p.H;
  const int k0 = kt * ROWS;
  const int j0 = k0 + warp * kWarpRows + 4 * ty;  // the lane's keys j0 .. j0 + 3
  const long long base = (long long)b * p.sB + (long long)h * p.sH;
  const TI* Q = reinterpret_cast<const TI*>(p.q) + base;
  const TI* K = reinterpret_cast<const TI*>(p.k) + base;
  const TI* V = reinterpret_cast<const TI*>(p.v) + base;
  const TI* G = reinterpret_cast<const TI*>(p.dout) + base;
  const float* logz = p.logz_in + (long long)bh * p.T;
  const float* Drow = ws.D + (long long)bh * p.T;
  const float* Fs = ws.F_self + (long long)bh * p.T;

  float dk[4][D / 16], dv[4][D / 16];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < D / 16; ++c) dk[r][c] = dv[r][c] = 0.f;
  Sum2 dlam;  // -sum_i log i F_ii dR_ij over the lane's Exchange pairs (they cancel within a row)
  stage<TI, D, NT * NG>(Ks, K, p.sT, k0, ROWS, p.T, threadIdx.x);
  stage<TI, D, NT * NG>(Vs, V, p.sT, k0, ROWS, p.T, threadIdx.x);
  if (NG > 1) {  // both groups read all of them
    stage_commit();
    stage_wait<0>();
    __syncthreads();
  }
  for (int q0 = k0 / kTile * kTile + grp * kTile; q0 < p.T; q0 += NG * kTile) {
    group_sync<NT, NG>(grp);  // the previous tile has been read
    stage<TI, D, NT>(Qs, Q, p.sT, q0, kTile, p.T, tid);
    stage<TI, D, NT>(Gs, G, p.sT, q0, kTile, p.T, tid);
    stage_commit();
    for (int ii = tid; ii < kTile; ii += NT) {
      const int i = q0 + ii;
      if (i < p.T) {
        // cs rounds; its error times P is in every P of the row, and taken out of dlambda's weight
        Sum2 c;
        c.add_log((float)(i + 1), -p.lambda);
        c.add(-logz[i]);
        cs[ii] = c.s;
        wl[ii] = logf((float)(i + 1)) * Fs[i] * (fabsf(c.s) < INFINITY ? 1.f + c.c : 1.f);
        Ds[ii] = Drow[i];
      } else {
        cs[ii] = -INFINITY;
        wl[ii] = Ds[ii] = 0.f;
      }
    }
    stage_wait<0>();
    group_sync<NT, NG>(grp);
    float P[4][4], dS[4][4];
    dots<D>(Ks + warp * kWarpRows * LD, Qs, ty, tx, P);
    dots<D>(Vs + warp * kWarpRows * LD, Gs, ty, tx, dS);
    float dl = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int ii = 16 * i + tx, q = q0 + ii;
      const float ci = cs[ii], Di = Ds[ii], wi = wl[ii];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float pv, dR, ds;
        pair_grad(P[r][i] * p.inv_sqrt_d, dS[r][i], ci, Di, pv, dR, ds);
        const bool in = q > j0 + r && q < p.T;
        P[r][i] = in ? pv : 0.f;
        dS[r][i] = in ? ds : 0.f;
        dl = in ? fmaf(-wi, dR, dl) : dl;
        Pw[(4 * ty + r) * PW + ii] = P[r][i];
      }
    }
    dlam.add(dl);
    __syncwarp();
    // queries after every key of the warp, and before them the (at most 8) mixed ones
    const int first = k0 + warp * kWarpRows + 1 - q0;  // the first query any key takes
    const int some = max(0, min(kTile, first & ~3));
    const int full = max(0, min(kTile, (first + kWarpRows - 1 + 3) & ~3));
    auto use = [&](int r, int k) { return q0 + k > j0 + r; };
    axpys<D, true>(Pw, Gs, ty, tx, some, full, dv, use);
    axpys<D, false>(Pw, Gs, ty, tx, full, kTile, dv, use);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int r = 0; r < 4; ++r) Pw[(4 * ty + r) * PW + 16 * i + tx] = dS[r][i];
    __syncwarp();
    axpys<D, true>(Pw, Qs, ty, tx, some, full, dk, use);
    axpys<D, false>(Pw, Qs, ty, tx, full, kTile, dk, use);
  }
  // the CTA's dlambda partial
  double lsum = (double)dlam.s + (double)dlam.c;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if (lane == 0) red[threadIdx.x >> 5] = (float)lsum;
  if (NG > 1) {  // the second group's dK, dV through its own tiles
    float* const xs = Vs + (ROWS + 2 * kTile) * LD + (warp * kWarpRows + 4 * ty) * LD;
    if (grp == 1) {
      group_sync<NT, NG>(grp);  // the last tile has been read
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        store_cols<float, D>(xs + r * LD, tx, dk[r]);
        store_cols<float, D>(xs + (kTile + r) * LD, tx, dv[r]);
      }
    }
    __syncthreads();
    if (grp == 1) return;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float a[D / 16], b2[D / 16];
      load_cols<float, D>(xs + r * LD, tx, a);
      load_cols<float, D>(xs + (kTile + r) * LD, tx, b2);
#pragma unroll
      for (int c = 0; c < D / 16; ++c) {
        dk[r][c] += a[c];
        dv[r][c] += b2[c];
      }
    }
  } else {
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < W * NG; ++w) t += red[w];
    dlam_part[kt * (p.B * p.H) + bh] = t;
  }
  // Self terms of key j: dv_j += F_jj dO_j, dk_j += dS_jj q_j; then the 1/sqrt(d) of U.
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int j = j0 + r;
    if (j >= p.T) continue;
    const float fs = Fs[j], dss = ws.dS_self[(long long)bh * p.T + j];
    float qj[D / 16], gj[D / 16];
    load_cols<TI, D>(Q + (long long)j * p.sT, tx, qj);
    load_cols<TI, D>(G + (long long)j * p.sT, tx, gj);
#pragma unroll
    for (int c = 0; c < D / 16; ++c) {
      qj[c] = (dk[r][c] + dss * qj[c]) * p.inv_sqrt_d;
      gj[c] = dv[r][c] + fs * gj[c];
    }
    store_cols<TI, D>(reinterpret_cast<TI*>(p.dk) + base + (long long)j * p.sT, tx, qj);
    store_cols<TI, D>(reinterpret_cast<TI*>(p.dv) + base + (long long)j * p.sT, tx, gj);
  }
}

// dQ (query-stationary): the CTA's ROWS queries over the key tiles up to its last query
template <typename TI, int D, int W, int NG>
__device__ __forceinline__ void bwd_dq(const Problem& p, const BwdWorkspace& ws, float* smem,
                                       int qt, int bh) {
  constexpr int LD = Ld<D>::V, ROWS = kWarpRows * W, NT = 32 * W;
  float* Qs = smem;
  float* Gs = Qs + ROWS * LD;
  const int grp = NG == 1 ? 0 : threadIdx.x / NT, tid = NG == 1 ? threadIdx.x : threadIdx.x % NT;
  float* Ks = Gs + ROWS * LD + grp * 2 * kTile * LD;
  float* Vs = Ks + kTile * LD;
  const int warp = tid >> 5, lane = tid & 31, ty = lane >> 4, tx = lane & 15;
  float* Pw = Gs + (ROWS + NG * 2 * kTile) * LD + (threadIdx.x >> 5) * kWarpRows * PW;
  const int b = bh / p.H, h = bh % p.H;
  const int q0 = qt * ROWS;
  const int r0 = q0 + warp * kWarpRows + 4 * ty;  // the lane's queries r0 .. r0 + 3
  const long long base = (long long)b * p.sB + (long long)h * p.sH;
  const TI* Q = reinterpret_cast<const TI*>(p.q) + base;
  const TI* K = reinterpret_cast<const TI*>(p.k) + base;
  const TI* V = reinterpret_cast<const TI*>(p.v) + base;
  const TI* G = reinterpret_cast<const TI*>(p.dout) + base;

  float dq[4][D / 16], ci[4], Di[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = r0 + r;
    const long long row = (long long)bh * p.T + min(i, p.T - 1);
    ci[r] = -p.lambda * logf((float)(i + 1)) - p.logz_in[row];
    Di[r] = ws.D[row];
#pragma unroll
    for (int c = 0; c < D / 16; ++c) dq[r][c] = 0.f;
  }
  const int kend = min(p.T, q0 + ROWS);
  constexpr int STEP = NG * kTile;
  stage<TI, D, NT * NG>(Qs, Q, p.sT, q0, ROWS, p.T, threadIdx.x);
  stage<TI, D, NT * NG>(Gs, G, p.sT, q0, ROWS, p.T, threadIdx.x);
  if (grp * kTile < kend) stage<TI, D, NT>(Vs, V, p.sT, grp * kTile, kTile, p.T, tid);
  stage_commit();
  if (NG > 1) {  // both groups read all of Q and dO
    stage_wait<0>();
    __syncthreads();
  }
  for (int k0 = grp * kTile; k0 < kend; k0 += STEP) {
    stage<TI, D, NT>(Ks, K, p.sT, k0, kTile, p.T, tid);
    stage_commit();
    stage_wait<1>();
    group_sync<NT, NG>(grp);  // V (and Q, dO) are in
    float dS[4][4], u[4][4];
    dots<D>(Gs + warp * kWarpRows * LD, Vs, ty, tx, dS);
    stage_wait<0>();
    group_sync<NT, NG>(grp);  // V has been read, K is in
    if (k0 + STEP < kend) stage<TI, D, NT>(Vs, V, p.sT, k0 + STEP, kTile, p.T, tid);
    stage_commit();
    dots<D>(Qs + warp * kWarpRows * LD, Ks, ty, tx, u);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float P, dR, ds;
        pair_grad(u[r][i] * p.inv_sqrt_d, dS[r][i], ci[r], Di[r], P, dR, ds);
        dS[r][i] = k0 + 16 * i + tx < r0 + r ? ds : 0.f;
        Pw[(4 * ty + r) * PW + 16 * i + tx] = dS[r][i];
      }
    __syncwarp();
    const int hist = q0 + warp * kWarpRows + kWarpRows - 1 - k0;
    const int full = max(0, min(kTile, (hist - kWarpRows + 1) & ~3));
    const int some = max(0, min(kTile, (hist + 3) & ~3));
    axpys<D, false>(Pw, Ks, ty, tx, 0, full, dq, [](int, int) { return true; });
    axpys<D, true>(Pw, Ks, ty, tx, full, some, dq, [&](int r, int k) { return k0 + k < r0 + r; });
    group_sync<NT, NG>(grp);  // K has been read
  }
  if (NG > 1) {  // the second group's dQ through its own tiles
    float* const xs = Gs + (ROWS + 2 * kTile) * LD + (warp * kWarpRows + 4 * ty) * LD;
    if (grp == 1) {
#pragma unroll
      for (int r = 0; r < 4; ++r) store_cols<float, D>(xs + r * LD, tx, dq[r]);
    }
    __syncthreads();
    if (grp == 1) return;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float a[D / 16];
      load_cols<float, D>(xs + r * LD, tx, a);
#pragma unroll
      for (int c = 0; c < D / 16; ++c) dq[r][c] += a[c];
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = r0 + r;
    if (i >= p.T) continue;
    const float dss = ws.dS_self[(long long)bh * p.T + i];
    float ki[D / 16];
    load_cols<TI, D>(K + (long long)i * p.sT, tx, ki);
#pragma unroll
    for (int c = 0; c < D / 16; ++c) ki[c] = (dq[r][c] + dss * ki[c]) * p.inv_sqrt_d;
    store_cols<TI, D>(reinterpret_cast<TI*>(p.dq) + base + (long long)i * p.sT, tx, ki);
  }
}

// Even CTAs dK / dV, odd ones dQ, the longest first in both.
template <typename TI, int D, int W, int NG>
__global__ void __launch_bounds__(32 * W * NG, NG == 2 && D < 128 ? 2 : 0) bwd_kernel(Problem p, BwdWorkspace ws, float* dlam_part,
                                                     int n_t) {
  extern __shared__ float4 smem_f4[];
  float* smem = reinterpret_cast<float*>(smem_f4);
  const int BH = p.B * p.H;
  const int t = (int)((blockIdx.x >> 1) / BH), bh = (int)((blockIdx.x >> 1) % BH);
  pdl_wait();
  if (blockIdx.x & 1)
    bwd_dq<TI, D, W, NG>(p, ws, smem, n_t - 1 - t, bh);
  else
    bwd_dkdv<TI, D, W, NG>(p, ws, dlam_part, smem, t, bh);
}

// dQ in the place of Q or dO, which the dK / dV CTAs of every earlier key read: a launch of its own
// behind theirs.  (A kernel for each: a switch in bwd_kernel costs it registers, 20 % at d 32.)
template <typename TI, int D, int W, bool DQ>
__global__ void __launch_bounds__(32 * W) bwd_part_kernel(Problem p, BwdWorkspace ws, float* dlam_part, int n_t) {
  extern __shared__ float4 smem_f4[];
  const int BH = p.B * p.H, t = (int)(blockIdx.x / BH), bh = (int)(blockIdx.x % BH);
  pdl_wait();
  if (DQ)
    bwd_dq<TI, D, W, 1>(p, ws, reinterpret_cast<float*>(smem_f4), n_t - 1 - t, bh);
  else
    bwd_dkdv<TI, D, W, 1>(p, ws, dlam_part, reinterpret_cast<float*>(smem_f4), t, bh);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
bool supports(relation_dtype dt, int d) {
  (void)dt;
  return d == 32 || d == 64 || d == 128;
}

// Warps per CTA (8 rows each).  Forward / backward tiles in us with 4 and with 2 warps: B 2,
// H 8, T 1000, d 64: 107 / 209, 104 / 239; B 2, H 4, T 777, d 128: 95 / 175, 92 / 194; B 4, H 8,
// T 1500, d 32: 189 / 520, 201 / 585; at T 128 alike.  Eight warps, both with IEEE division in
// the sigmoid: 134 / 236 against 127 / 222, 150 / 215 against 130 / 195, 251 / 586 against
// 228 / 566.
constexpr int kWarps = 4;

static int tiles(const Problem& p) {
  return (p.T + kWarpRows * kWarps - 1) / (kWarpRows * kWarps);
}

// Two groups per CTA where the longest row's chain of tiles decides, which it does up to some number
// of CTAs per SM.  Beyond it two groups only cost residency (at d 64 two of their CTAs fit an SM, for
// four (forward) and three (backward) of one group; at d 128 one for two), registers and the
// joining.  The lines are where both forms take the same time, measured with each forced, and lie
// lower up to 128 tokens: two tiles, little to share.  us with one and with two groups, below the
// line and above it (B H, T):
//   forward, d <= 64:  T <= 128, 2 per SM: 64, 128 14.0 / 12.9, 96, 128 17.0 / 21.5;
//                      longer, 4: 16, 1000 98 / 81, 48, 500 59 / 68
//   forward, d 128:    1: 32, 128 17.0 / 15.4, 48, 128 19.3 / 23.9; 2: 16, 500 61 / 53, 24, 500 67 / 76
//   backward, d <= 64: 3: 48, 128 33.1 / 28.4, 64, 128 34.5 / 34.4; 5: 12, 777 161 / 117,
//                      16, 1000 210 / 218
//   backward, d 128:   2: 32, 128 40.0 / 35.7, 48, 128 40.5 / 47.1; 3: 8, 777 197 / 148,
//                      16, 640 168 / 185
static bool two_groups(const Problem& p, long long ctas, int short_per_sm, int per_sm) {
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    nsm = 0;
  return p.T > kTile && ctas <= (long long)(p.T > 2 * kTile ? per_sm : short_per_sm) * nsm;
}

template <typename TI, int D, int NG>
static cudaError_t fwd_g(const Problem& p, unsigned grid, cudaStream_t s) {
  constexpr int W = kWarps;
  constexpr size_t smem = fwd_smem<D, W, NG>();
  static_assert(smem <= 232448, "shared memory");
  const cudaError_t e = cudaFuncSetAttribute(
      fwd_kernel<TI, D, W, NG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(fwd_kernel<TI, D, W, NG>, dim3(grid), 32 * W * NG, smem, s, 1, p, tiles(p));
}

template <typename TI, int D, int NG>
static cudaError_t bwd_g(const Problem& p, const BwdWorkspace& ws, unsigned grid, cudaStream_t s) {
  constexpr int W = kWarps;
  constexpr size_t smem = bwd_smem<D, W, NG>();
  static_assert(smem <= 232448, "shared memory");
  const cudaError_t e = cudaFuncSetAttribute(
      bwd_kernel<TI, D, W, NG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(bwd_kernel<TI, D, W, NG>, dim3(grid), 32 * W * NG, smem, s, 1, p, ws,
                    main_partials(ws), tiles(p));
}

template <typename TI, int D, bool DQ>
static cudaError_t bwd_part(const Problem& p, const BwdWorkspace& ws, unsigned grid, cudaStream_t s) {
  constexpr int W = kWarps;
  constexpr size_t smem = bwd_smem<D, W, 1>();
  const cudaError_t e = cudaFuncSetAttribute(
      bwd_part_kernel<TI, D, W, DQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(bwd_part_kernel<TI, D, W, DQ>, dim3(grid), 32 * W, smem, s, 1, p, ws,
                    main_partials(ws), tiles(p));
}

template <typename TI, int D>
static cudaError_t fwd_t(const Problem& p, cudaStream_t s) {
  const long long grid = (long long)tiles(p) * p.B * p.H;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  return two_groups(p, grid, D < 128 ? 2 : 1, D < 128 ? 4 : 2) ? fwd_g<TI, D, 2>(p, (unsigned)grid, s)
                             : fwd_g<TI, D, 1>(p, (unsigned)grid, s);
}

template <typename TI, int D>
static cudaError_t bwd_t(const Problem& p, const BwdWorkspace& ws, cudaStream_t s) {
  const long long grid = 2LL * tiles(p) * p.B * p.H;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  if (p.dq == p.q || p.dq == p.dout) {
    const cudaError_t e = bwd_part<TI, D, false>(p, ws, (unsigned)(grid / 2), s);
    return e != cudaSuccess ? e : bwd_part<TI, D, true>(p, ws, (unsigned)(grid / 2), s);
  }
  return two_groups(p, grid, D < 128 ? 3 : 2, D < 128 ? 5 : 3) ? bwd_g<TI, D, 2>(p, ws, (unsigned)grid, s)
                             : bwd_g<TI, D, 1>(p, ws, (unsigned)grid, s);
}

// The tile kernel's dlambda partials, one per dK / dV CTA and its 32 rows: in the tensor-core path's
// per-query scalars (four floats per row, rows padded to 128), which this path does not use.
static_assert(128 % (kWarpRows * kWarps) == 0, "a head's partials end within its padded rows");
float* main_partials(const BwdWorkspace& ws) { return ws.stats; }
int main_ctas(const Problem& p) { return tiles(p) * p.B * p.H; }

template <int D>
static cudaError_t fwd_d(const Problem& p, cudaStream_t s) {
  return p.dtype == RELATION_F32 ? fwd_t<float, D>(p, s) : fwd_t<__nv_bfloat16, D>(p, s);
}
template <int D>
static cudaError_t bwd_d(const Problem& p, const BwdWorkspace& ws, cudaStream_t s) {
  return p.dtype == RELATION_F32 ? bwd_t<float, D>(p, ws, s) : bwd_t<__nv_bfloat16, D>(p, ws, s);
}

cudaError_t launch_fwd(const Problem& p, cudaStream_t s) {
  switch (p.d) {
    case 32: return fwd_d<32>(p, s);
    case 64: return fwd_d<64>(p, s);
    case 128: return fwd_d<128>(p, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_bwd(const Problem& p, const BwdWorkspace& ws, cudaStream_t s) {
  switch (p.d) {
    case 32: return bwd_d<32>(p, ws, s);
    case 64: return bwd_d<64>(p, ws, s);
    case 128: return bwd_d<128>(p, ws, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace simt
}  // namespace rel
