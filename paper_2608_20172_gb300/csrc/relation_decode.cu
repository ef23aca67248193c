// relation_decode.cu -- one new token per sequence against a key/value cache.
//
// Decoding with the causal Relation operator (Sec. 3.1; the factorised row of Sec. 4.2 /
// App. A.1): sequence b of the batch holds len_b cached rows whose last row is the new
// token, at one-based position i = len_b.  Per (b, h):
//   Exchange over the history j < i (cache rows 0 .. len_b - 2):
//       E_j = SiLU(q . k_j / sqrt(d)),  L^E = log sum_j e^{E_j},  z = sum_j e^{E_j} v_j
//   Self (cache row len_b - 1):  S = sigmoid(q . k_i / (sqrt(d) tau_S))
//   A = L^E - lambda log i,  g = sigmoid(A - S),  Y = (1 - g) v_i + g z / sum_j e^{E_j},
//   logZ = logaddexp(S, A);  a one-row cache (i = 1) has no history: g = 0, Y = v_1,
//   logZ = S.
// This is the last row of the full forward over the cache, evaluated without the other
// rows.  Memory-bound: every cached key and value is read once.
//
// Few heads, short caches: one launch, a cluster of CTAs per head, each with its share of the
// history; the CTAs leave (m, l, z) = (max E, sum e^{E - m}, sum e^{E - m} v) in their shared
// memory and the first merges them through distributed shared memory and applies the
// Self-Exchange epilogue.  There the time is latency: launches, and dependent trips to memory.
// Otherwise two launches: the partial pass splits each history into chunks of kChunk rows, one
// CTA per (head, chunk), with (m, l, z) to the workspace; the combine pass (one CTA per head)
// merges them by the associative (m, l, z) rule of the tiled scan (App. A.3), the chunks' weights
// a thread each (a serial loop over dependent loads before).  It starts when the partial pass has
// ended: CTAs that come in early (pdl_launch) cost a grid of 512 heads 0.7 to 1.7 us and gain
// nothing elsewhere.
// Measured in one graph over caches that together exceed L2, bf16, before -> now:
// B 1, H 12, T 2048, d 64 18.6 -> 8.7 us; B 1, H 32, T 2048, d 80 78 -> 13.6;
// B 32, H 8, T 2048, d 80 148 -> 54.8; B 1, H 16, T 32768, d 128 92.7 -> 56.6 (68.2 with the merge's
// loads one behind the other); B 32, H 16, T 8192, d 128 (2.1 GB) 331 -> 319 (6.74 TB/s).
#include <cooperative_groups.h>
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace rel {
namespace decode {

namespace cg = cooperative_groups;

constexpr int kChunk = 512;   // history rows of a partial (m, l, z)
constexpr int kWarps = 8;      // of a partial CTA
constexpr int kMaxD = 128;
constexpr int kCluster = 8;    // CTAs per head where the heads are few,
constexpr int kClWarps = 4;    // their warps,
constexpr int kClStages = 2;   // and a warp's tiles in flight

template <typename TI>
__device__ __forceinline__ float ldf(const TI* p);
template <>
__device__ __forceinline__ float ldf<float>(const float* p) { return __ldg(p); }
template <>
__device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(*p);
}

// 16 bytes of a row as fp32
template <typename TI>
struct Vec;
template <>
struct Vec<float> {
  static constexpr int N = 4;
  static __device__ __forceinline__ void unpack(const uint4& w, float (&x)[4]) {
    x[0] = __uint_as_float(w.x); x[1] = __uint_as_float(w.y);
    x[2] = __uint_as_float(w.z); x[3] = __uint_as_float(w.w);
  }
};
template <>
struct Vec<__nv_bfloat16> {
  static constexpr int N = 8;
  static __device__ __forceinline__ void unpack(const uint4& w, float (&x)[8]) {
    const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&ww[e]));
      x[2 * e] = f.x; x[2 * e + 1] = f.y;
    }
  }
};
// 16 bytes to shared memory, zeros if not ok
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src),
               "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ float silu(float u) { return u / (1.0f + expf(-u)); }

__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// A cluster CTA's shared memory beside its ring
struct Smem {
  float p[kClWarps][32];      // a warp's tile of weights
  float zs[kClWarps][32 * 8], ms[kClWarps], ls[kClWarps];  // the warps' (z, m, l)
  float m, l, z[kMaxD];       // the CTA's
  float self;                 // q . k_i
};

// One warp's part of the (m, l, z) of a run of cache rows.  Every warp keeps its own (m, l, z)
// over tiles of rows, so that nothing waits for another warp before the run's end.
// NQ > 0: rows in 16-byte groups (aligned, d a multiple of Vec::N, at most 4 NQ groups); scores
// with four lanes per key (lane & 3 takes the groups lane & 3, + 4, ...), P V with a lane per
// group and 32 / groups rows at once.  A lane's 8 groups of a tile's keys and 8 of its values
// come by cp.async, S tiles ahead of their use, into shared memory that it alone writes and
// reads.  NQ = 0: any d <= 128 and alignment, a lane per column, 32 at a time, plain loads.
template <typename TI, int NQ>
struct Scan {
  static constexpr int W = kClWarps, S = kClStages;
  static constexpr int NE = NQ > 0 ? Vec<TI>::N : 4;  // elements of z per lane
  static constexpr int KR = NQ > 0 ? 8 / NQ : 1;      // keys per lane
  static constexpr int KT = NQ > 0 ? 8 * KR : 4;      // keys per tile
  static constexpr int NR = NQ > 0 ? NQ : 1;
  static constexpr int kRing = NQ > 0 ? W * S * 16 * 32 * 16 : 0;  // bytes of a CTA's ring
  const DecodeProblem& p;
  Smem& sm;
  const uint4* ring;  // this lane's first slot
  int warp, lane, nv, G, g, u;
  float q[NR][NE], m, l, z[NE];

  __device__ __forceinline__ Scan(const DecodeProblem& p, Smem& sm, const uint4* smem_ring)
      : p(p), sm(sm) {
    warp = threadIdx.x >> 5;
    lane = threadIdx.x & 31;
    ring = smem_ring + warp * S * 16 * 32 + lane;
    nv = NQ > 0 ? p.d / NE : 32;  // groups of a row
    G = 32 / nv;                  // rows per load of the values
    g = lane / nv;
    u = lane - g * nv;
  }
  __device__ __forceinline__ void start(const TI* qv) {
#pragma unroll
    for (int t = 0; t < NR; ++t)
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        const int c = NQ > 0 ? ((lane & 3) + 4 * t) * NE + e : lane + 32 * e;
        q[t][e] = c < p.d ? ldf<TI>(qv + c) : 0.f;
      }
    m = -INFINITY;
    l = 0.f;
#pragma unroll
    for (int e = 0; e < NE; ++e) z[e] = 0.f;
  }
  // a tile's largest E exceeds m: rescale (-inf: nothing yet)
  __device__ __forceinline__ void raise(float mx) {
    const float mn = fmaxf(m, mx), sc = m == -INFINITY ? 0.f : expf(m - mn);
    m = mn;
    l *= sc;
#pragma unroll
    for (int e = 0; e < NE; ++e) z[e] *= sc;
  }
  // rows j .. j + KT - 1 of the n from kc, vc to stage st (rows past n: zeros)
  __device__ __forceinline__ void fetch(const TI* kc, const TI* vc, int n, int j, int st) {
    const uint32_t dst = smem_u32(ring + st * 16 * 32);
    const int sub = lane & 3, slot = lane >> 2;
#pragma unroll
    for (int r = 0; r < KR; ++r) {
      const bool in = j + 8 * r + slot < n;
      const TI* row = kc + (long long)(in ? j + 8 * r + slot : 0) * p.sT;
#pragma unroll
      for (int t = 0; t < NR; ++t) {
        const bool ok = in && sub + 4 * t < nv;
        cp16(dst + (r * NR + t) * 512, row + (ok ? (sub + 4 * t) * NE : 0), ok);
      }
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int i = t * G + g;
      const bool ok = g < G && i < KT && j + i < n;
      cp16(dst + (8 + t) * 512, vc + (ok ? (long long)(j + i) * p.sT + u * NE : 0), ok);
    }
  }
  // the tile in stage st
  __device__ __forceinline__ void tile(int n, int j, int st) {
    const uint4* in = ring + st * 16 * 32;
    const int sub = lane & 3, slot = lane >> 2;
    float E[KR], mx = -INFINITY;
#pragma unroll
    for (int r = 0; r < KR; ++r) {
      float s = 0.f;
#pragma unroll
      for (int t = 0; t < NR; ++t) {
        float x[NE];
        Vec<TI>::unpack(in[(r * NR + t) * 32], x);
#pragma unroll
        for (int e = 0; e < NE; ++e) s = fmaf(q[t][e], x[e], s);
      }
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      E[r] = silu(s * p.inv_sqrt_d);
      if (j + 8 * r + slot < n) mx = fmaxf(mx, E[r]);
    }
    if (__any_sync(0xffffffffu, mx > m)) raise(warp_max(mx));
#pragma unroll
    for (int r = 0; r < KR; ++r) {
      const float P = j + 8 * r + slot < n ? expf(E[r] - m) : 0.f;
      if (sub == 0) {
        sm.p[warp][8 * r + slot] = P;
        l += P;
      }
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const float P = sm.p[warp][min(t * G + g, KT - 1)];  // (past the tile: times zeros)
      float x[NE];
      Vec<TI>::unpack(in[(8 + t) * 32], x);
#pragma unroll
      for (int e = 0; e < NE; ++e) z[e] = fmaf(P, x[e], z[e]);
    }
    __syncwarp();  // sm.p is written again
  }
  // NQ = 0: the rows j .. j + KT - 1 by plain loads
  __device__ __forceinline__ void tile_plain(const TI* kc, const TI* vc, int n, int j) {
    float x[KT][NE], y[KT][NE], E[KT], mx = -INFINITY;
#pragma unroll
    for (int r = 0; r < KT; ++r)
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        const bool in = j + r < n && lane + 32 * e < p.d;
        const long long at = (long long)(j + r) * p.sT + lane + 32 * e;
        x[r][e] = in ? ldf<TI>(kc + at) : 0.f;
        y[r][e] = in ? ldf<TI>(vc + at) : 0.f;
      }
#pragma unroll
    for (int r = 0; r < KT; ++r) {
      float s = 0.f;
#pragma unroll
      for (int e = 0; e < NE; ++e) s = fmaf(q[0][e], x[r][e], s);
      E[r] = silu(warp_sum(s) * p.inv_sqrt_d);
      if (j + r < n) mx = fmaxf(mx, E[r]);
    }
    if (mx > m) raise(mx);
#pragma unroll
    for (int r = 0; r < KT; ++r) {
      const float P = j + r < n ? expf(E[r] - m) : 0.f;
      l += P;
#pragma unroll
      for (int e = 0; e < NE; ++e) z[e] = fmaf(P, y[r][e], z[e]);
    }
  }
  // this warp's tiles of the n rows from kc, vc
  __device__ __forceinline__ void run(const TI* qv, const TI* kc, const TI* vc, int n) {
    const int j0 = warp * KT;
    if constexpr (NQ > 0) {
#pragma unroll
      for (int st = 0; st < S; ++st) {
        if (j0 + st * W * KT < n) fetch(kc, vc, n, j0 + st * W * KT, st);
        cp_commit();
      }
    }
    start(qv);
    int st = 0;
    for (int j = j0; j < n; j += W * KT) {
      if constexpr (NQ > 0) {
        cp_wait<S - 1>();
        tile(n, j, st);
        if (j + S * W * KT < n) fetch(kc, vc, n, j + S * W * KT, st);
        cp_commit();
        st = st + 1 == S ? 0 : st + 1;
      } else {
        tile_plain(kc, vc, n, j);
      }
    }
  }
  // merge the warps (and a warp's row groups): *om, *ol and oz[0 .. d) by the CTA's threads
  __device__ __forceinline__ void merge(float* om, float* ol, float* oz) {
    if (NQ > 0) l = warp_sum(l);
    if (lane == 0) {
      sm.ms[warp] = m;
      sm.ls[warp] = l;
    }
#pragma unroll
    for (int e = 0; e < NE; ++e) sm.zs[warp][NQ > 0 ? lane * NE + e : lane + 32 * e] = z[e];
    __syncthreads();
    const int c = threadIdx.x;
    if (c >= p.d) return;
    float M = -INFINITY, L = 0.f, Z = 0.f;
#pragma unroll
    for (int w = 0; w < W; ++w) M = fmaxf(M, sm.ms[w]);
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const float a = sm.ms[w] == -INFINITY ? 0.f : expf(sm.ms[w] - M);
      L = fmaf(a, sm.ls[w], L);
      float zt = 0.f;
      for (int k = 0; k < G; ++k) zt += sm.zs[w][k * p.d + c];
      Z = fmaf(a, zt, Z);
    }
    oz[c] = Z;
    if (c == 0) {
      *om = M;  // -inf without history
      *ol = L;  // 0 without history
    }
  }
};

// Self evidence q . k_i by one warp
template <typename TI>
__device__ __forceinline__ float self_dot(const DecodeProblem& p, const TI* qv, const TI* ks,
                                          int lane) {
  float s = 0.f;
  for (int c = lane; c < p.d; c += 32) s = fmaf(ldf<TI>(qv + c), ldf<TI>(ks + c), s);
  return warp_sum(s);
}

// Column c of the new row from the merged (M, L, Z): the Self-Exchange epilogue
template <typename TI>
__device__ __forceinline__ void epilogue(const DecodeProblem& p, int bh, int len, float qk, float M,
                                         float L, float Z, int c, float vi, TI* o) {
  const float S = 1.0f / (1.0f + expf(-(qk * p.inv_sqrt_d) / p.tau_s));
  float g = 0.f, lz = S, fz = 0.f;
  if (len > 1 && L > 0.f) {
    const float A = M + logf(L) - p.lambda * logf((float)len);
    g = 1.0f / (1.0f + expf(S - A));
    const float hi = fmaxf(S, A), lo = fminf(S, A);
    lz = hi + log1pf(expf(lo - hi));
    fz = Z / L;
  }
  const float y = fmaf(g, fz - vi, vi);
  if (sizeof(TI) == 4)
    reinterpret_cast<float*>(o)[c] = y;
  else
    reinterpret_cast<__nv_bfloat16*>(o)[c] = __float2bfloat16_rn(y);
  if (c == 0) p.logz[bh] = lz;
}

// A sequence's length, 0 (reported) where it lies outside [1, T]
__device__ __forceinline__ int length_of(const DecodeProblem& p, int b, bool report) {
  const int len = p.lengths[b];
  if (len >= 1 && len <= p.T) return len;
  if (report && p.dev_status) atomicExch(p.dev_status, (int)RELATION_ERR_INVALID_ARG);
  return 0;
}

// One cluster per head.  The cluster's CTAs meet twice whatever the length.
template <typename TI, int NQ>
__global__ void __launch_bounds__(32 * kClWarps) cluster_kernel(DecodeProblem p) {
  using SC = Scan<TI, NQ>;
  constexpr int W = kClWarps;
  __shared__ Smem sm;
  extern __shared__ uint4 ring[];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)blockIdx.x % kCluster;
  const int bh = (int)blockIdx.x / kCluster, b = bh / p.H, h = bh % p.H;
  pdl_wait_and_launch();
  const int len = length_of(p, b, threadIdx.x == 0 && rank == 0);
  const TI* qv = reinterpret_cast<const TI*>(p.q) + (long long)b * p.qsB + (long long)h * p.qsH;
  const long long head = (long long)b * p.sB + (long long)h * p.sH;
  const TI* kh = reinterpret_cast<const TI*>(p.k) + head;
  const TI* vh = reinterpret_cast<const TI*>(p.v) + head;
  if (len > 0) {
    const int hist = len - 1, per = (hist + kCluster - 1) / kCluster;
    const int r0 = min(hist, rank * per), n = min(per, hist - r0);
    const TI* kc = kh + (long long)r0 * p.sT;
    const TI* vc = vh + (long long)r0 * p.sT;
    SC sc(p, sm, ring);
    sc.run(qv, kc, vc, n);
    if (rank == 0 && sc.warp == W - 1) {
      const float s = self_dot<TI>(p, qv, kh + (long long)(len - 1) * p.sT, sc.lane);
      if (sc.lane == 0) sm.self = s;
    }
    sc.merge(&sm.m, &sm.l, sm.z);
  }
  cl.sync();
  const int c = threadIdx.x;
  if (rank == 0 && len > 0 && c < p.d) {
    float mr[kCluster], M = -INFINITY, L = 0.f, Z = 0.f;
#pragma unroll
    for (int r = 0; r < kCluster; ++r) {
      mr[r] = *cl.map_shared_rank(&sm.m, r);
      M = fmaxf(M, mr[r]);
    }
#pragma unroll
    for (int r = 0; r < kCluster; ++r) {
      const Smem* o = cl.map_shared_rank(&sm, r);
      const float w = mr[r] == -INFINITY ? 0.f : expf(mr[r] - M);
      L = fmaf(w, o->l, L);
      Z = fmaf(w, o->z[c], Z);
    }
    epilogue<TI>(p, bh, len, sm.self, M, L, Z, c, ldf<TI>(vh + (long long)(len - 1) * p.sT + c),
                 reinterpret_cast<TI*>(p.out) + (long long)b * p.qsB + (long long)h * p.qsH);
  }
  cl.sync();  // the other CTAs' shared memory has been read
}

// Loads of n consecutive elements as fp32 (n * sizeof(TI) is 4, 8 or 16 bytes, aligned).
template <typename TI, int N>
__device__ __forceinline__ void ld_vec(const TI* p, float* out) {
  if constexpr (sizeof(TI) == 4) {
    static_assert(N % 4 == 0 || N <= 2, "fp32 vector width");
    if constexpr (N == 1) {
      out[0] = __ldg(reinterpret_cast<const float*>(p));
    } else if constexpr (N == 2) {
      const float2 v = __ldg(reinterpret_cast<const float2*>(p));
      out[0] = v.x; out[1] = v.y;
    } else {
#pragma unroll
      for (int i = 0; i < N; i += 4) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p + i));
        out[i] = v.x; out[i + 1] = v.y; out[i + 2] = v.z; out[i + 3] = v.w;
      }
    }
  } else {
    if constexpr (N == 2) {
      const uint32_t w = __ldg(reinterpret_cast<const unsigned int*>(p));
      const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w));
      out[0] = f.x; out[1] = f.y;
    } else if constexpr (N == 4) {
      const uint2 w = __ldg(reinterpret_cast<const uint2*>(p));
      const uint32_t ww[2] = {w.x, w.y};
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&ww[e]));
        out[2 * e] = f.x; out[2 * e + 1] = f.y;
      }
    } else {
      static_assert(N % 8 == 0, "bf16 vector width");
#pragma unroll
      for (int i = 0; i < N; i += 8) {
        const uint4 w = __ldg(reinterpret_cast<const uint4*>(p + i));
        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&ww[e]));
          out[i + 2 * e] = f.x; out[i + 2 * e + 1] = f.y;
        }
      }
    }
  }
}

// Partial (m, l, z) of history rows [c0, min(c0 + kChunk, len - 1)) of head (b, h), into part.
// Aligned rows of any whole number of 16-byte groups:
template <typename TI, int NQ>
__global__ void __launch_bounds__(32 * kClWarps) scan_kernel(DecodeProblem p, float* part) {
  __shared__ Smem sm;
  extern __shared__ uint4 ring[];
  pdl_wait();
  const int bh = blockIdx.x, chunk = blockIdx.y, b = bh / p.H, h = bh % p.H;
  const int len = length_of(p, b, threadIdx.x == 0 && chunk == 0);
  const int c0 = chunk * kChunk, n = min(kChunk, len - 1 - c0);
  if (n <= 0) return;  // (the combine pass reads only the chunks that hold history)
  const TI* qv = reinterpret_cast<const TI*>(p.q) + (long long)b * p.qsB + (long long)h * p.qsH;
  const long long at = (long long)b * p.sB + (long long)h * p.sH + (long long)c0 * p.sT;
  Scan<TI, NQ> sc(p, sm, ring);
  sc.run(qv, reinterpret_cast<const TI*>(p.k) + at, reinterpret_cast<const TI*>(p.v) + at, n);
  float* out = part + ((long long)bh * gridDim.y + chunk) * (2 + kMaxD);
  sc.merge(out, out + 1, out + 2);
}

// The same in two steps, the chunk's scores first, then P V.  D = 64 or 128 and aligned rows: four
// lanes per key and a quarter of the row each, then D / 32 consecutive columns per lane.  Fewer
// instructions per row than scan_kernel and twice the warps: where every SM is full, these bound
// the pass.  D = 0: any d and alignment, one element per lane and load, a warp per row; the warps
// keep many rows' loads in flight, where scan_kernel's plain loads wait tile by tile (bf16, d 64,
// rows of 65 elements, us with these and with those: 40 heads, T 300 18 / 31; 40 heads, T 4096
// 40 / 52; 512 heads, T 4096 269 / 315).
template <typename TI, int D>
__global__ void __launch_bounds__(32 * kWarps) partial_kernel(DecodeProblem p, float* part) {
  __shared__ float e_s[kChunk];
  __shared__ float red[kWarps];
  __shared__ float zs[kWarps][kMaxD];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.x, chunk = blockIdx.y;
  const int b = bh / p.H, h = bh % p.H;
  pdl_wait();
  int len;  // invalid (reported): no cache row is touched
  if constexpr (D > 0) {
    if ((len = length_of(p, b, threadIdx.x == 0 && chunk == 0)) == 0) return;
  } else {  // the same with the range in the compiler's sight: 40 registers in fp32 instead of 45,
            // 15 % of the pass
    len = p.lengths[b];
    if (len < 1 || len > p.T) {
      if (threadIdx.x == 0 && chunk == 0 && p.dev_status)
        atomicExch(p.dev_status, (int)RELATION_ERR_INVALID_ARG);
      return;
    }
  }
  const int hist = len - 1;  // history rows
  const int c0 = chunk * kChunk;
  const int n = max(0, min(kChunk, hist - c0));
  const TI* qv = reinterpret_cast<const TI*>(p.q) + (long long)b * p.qsB + (long long)h * p.qsH;
  const TI* kc = reinterpret_cast<const TI*>(p.k) + (long long)b * p.sB + (long long)h * p.sH +
                 (long long)c0 * p.sT;
  const TI* vc = reinterpret_cast<const TI*>(p.v) + (long long)b * p.sB + (long long)h * p.sH +
                 (long long)c0 * p.sT;
  constexpr int PL = D > 0 ? D / 32 : kMaxD / 32;  // columns per lane in the P V pass
  float mx = -INFINITY;
  if constexpr (D > 0) {
    // scores: lane = 4 key + quarter; per iteration two groups of 8 keys,
    // jj = base + lane / 4 and jj + 8 kWarps, loaded together (rows past the chunk read a
    // clamped row and are dropped)
    constexpr int QD = D / 4;
    const int sub = lane & 3, slot = lane >> 2;
    float qr[QD];
    ld_vec<TI, QD>(qv + sub * QD, qr);
    for (int base = warp * 8; base < n; base += 16 * kWarps) {
      const int j0 = base + slot, j1 = j0 + 8 * kWarps;
      float k0[QD], k1[QD];
      ld_vec<TI, QD>(kc + (long long)min(j0, n - 1) * p.sT + sub * QD, k0);
      ld_vec<TI, QD>(kc + (long long)min(j1, n - 1) * p.sT + sub * QD, k1);
      float s0 = 0.f, s1 = 0.f;
#pragma unroll
      for (int e = 0; e < QD; ++e) {
        s0 = fmaf(qr[e], k0[e], s0);
        s1 = fmaf(qr[e], k1[e], s1);
      }
      s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
      s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
      s0 += __shfl_xor_sync(0xffffffffu, s0, 2);
      s1 += __shfl_xor_sync(0xffffffffu, s1, 2);
      if (j0 < n) {
        const float u = s0 * p.inv_sqrt_d;
        const float E = u / (1.0f + expf(-u));  // SiLU(u)
        if (sub == 0) e_s[j0] = E;
        mx = fmaxf(mx, E);
      }
      if (j1 < n) {
        const float u = s1 * p.inv_sqrt_d;
        const float E = u / (1.0f + expf(-u));
        if (sub == 0) e_s[j1] = E;
        mx = fmaxf(mx, E);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  } else {
    float qr[PL];
#pragma unroll
    for (int e = 0; e < PL; ++e) {
      const int c = lane + 32 * e;
      qr[e] = c < p.d ? ldf<TI>(qv + c) : 0.f;
    }
    for (int jj = warp; jj < n; jj += kWarps) {
      const TI* kr = kc + (long long)jj * p.sT;
      float s = 0.f;
#pragma unroll
      for (int e = 0; e < PL; ++e) {
        const int c = lane + 32 * e;
        if (c < p.d) s = fmaf(qr[e], ldf<TI>(kr + c), s);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const float u = s * p.inv_sqrt_d;
      const float E = u / (1.0f + expf(-u));  // SiLU(u)
      if (lane == 0) e_s[jj] = E;
      mx = fmaxf(mx, E);
    }
  }
  if (lane == 0) red[warp] = mx;
  __syncthreads();
  float m = -INFINITY;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) m = fmaxf(m, red[w]);
  __syncthreads();
  // l = sum e^{E - m},  z = sum e^{E - m} v_j
  float l = 0.f, z[PL];
#pragma unroll
  for (int e = 0; e < PL; ++e) z[e] = 0.f;
  if constexpr (D > 0) {
    const int col = lane * PL;
#pragma unroll 8
    for (int jj = warp; jj < n; jj += kWarps) {
      const float P = expf(e_s[jj] - m);
      l += P;
      float vr[PL];
      ld_vec<TI, PL>(vc + (long long)jj * p.sT + col, vr);
#pragma unroll
      for (int e = 0; e < PL; ++e) z[e] = fmaf(P, vr[e], z[e]);
    }
#pragma unroll
    for (int e = 0; e < PL; ++e) zs[warp][col + e] = z[e];
  } else {
    for (int jj = warp; jj < n; jj += kWarps) {
      const float P = expf(e_s[jj] - m);
      l += P;
      const TI* vr = vc + (long long)jj * p.sT;
#pragma unroll
      for (int e = 0; e < PL; ++e) {
        const int c = lane + 32 * e;
        if (c < p.d) z[e] = fmaf(P, ldf<TI>(vr + c), z[e]);
      }
    }
#pragma unroll
    for (int e = 0; e < PL; ++e) zs[warp][lane + 32 * e] = z[e];
  }
  if (lane == 0) red[warp] = l;
  __syncthreads();
  float* out = part + ((long long)bh * gridDim.y + chunk) * (2 + kMaxD);
  if (threadIdx.x == 0) {
    float lt = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) lt += red[w];
    out[0] = m;   // -inf for an empty chunk
    out[1] = lt;  // 0 for an empty chunk
  }
  for (int c = threadIdx.x; c < p.d; c += blockDim.x) {
    float zt = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) zt += zs[w][c];
    out[2 + c] = zt;
  }
}

// Merge the chunks of head (b, h); thread c owns column c.
template <typename TI>
__global__ void __launch_bounds__(kMaxD) combine_kernel(DecodeProblem p, const float* part,
                                                        int n_chunks) {
  constexpr int kAhead = 16;  // chunks' z in flight
  __shared__ float red[kMaxD / 32], w[kMaxD], lw[kMaxD];
  __shared__ float self;
  const int bh = blockIdx.x, c = threadIdx.x, b = bh / p.H, h = bh % p.H;
  const int lane = c & 31, warp = c >> 5;
  // Before anything is read: that the partial CTAs have waited orders this kernel behind what came
  // before them, but only its own wait makes those writes visible here.
  pdl_wait_and_launch();
  const int len = length_of(p, b, false);  // (reported by the partial pass)
  if (len == 0) return;
  const TI* qv = reinterpret_cast<const TI*>(p.q) + (long long)b * p.qsB + (long long)h * p.qsH;
  const long long row = (long long)b * p.sB + (long long)h * p.sH + (long long)(len - 1) * p.sT;
  // the new row, in flight during the merge (K's by the last warp, which has no chunk weights to load)
  const bool own = warp == kMaxD / 32 - 1;
  float qr[kMaxD / 32], kr[kMaxD / 32];
#pragma unroll
  for (int e = 0; e < kMaxD / 32; ++e) {
    const bool in = own && lane + 32 * e < p.d;
    qr[e] = in ? ldf<TI>(qv + lane + 32 * e) : 0.f;
    kr[e] = in ? ldf<TI>(reinterpret_cast<const TI*>(p.k) + row + lane + 32 * e) : 0.f;
  }
  const float vi = c < p.d ? ldf<TI>(reinterpret_cast<const TI*>(p.v) + row + c) : 0.f;
  const int used = (len - 1 + kChunk - 1) / kChunk;  // <= n_chunks
  const float* pb = part + (long long)bh * n_chunks * (2 + kMaxD);
  float M = -INFINITY;
  for (int k = c; k < used; k += kMaxD) M = fmaxf(M, pb[(long long)k * (2 + kMaxD)]);
  M = warp_max(M);
  if (lane == 0) red[warp] = M;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kMaxD / 32; ++i) M = fmaxf(M, red[i]);
  if (own) {  // Self evidence q . k_i
    float s = 0.f;
#pragma unroll
    for (int e = 0; e < kMaxD / 32; ++e) s = fmaf(qr[e], kr[e], s);
    s = warp_sum(s);
    if (lane == 0) self = s;
  }
  float L = 0.f, Z = 0.f;
  for (int k0 = 0; k0 < used; k0 += kMaxD) {  // kMaxD chunks' weights at a time
    if (k0 > 0) __syncthreads();
    if (k0 + c < used) {
      const float* pk = pb + (long long)(k0 + c) * (2 + kMaxD);
      w[c] = pk[0] == -INFINITY ? 0.f : expf(pk[0] - M);
      lw[c] = pk[1];
    }
    __syncthreads();
    const int n = min(kMaxD, used - k0);
    for (int k = 0; k < n; k += kAhead) {  // (left to the unroller, the loads came one by one)
      float zk[kAhead];
#pragma unroll
      for (int e = 0; e < kAhead; ++e)
        zk[e] = k + e < n && c < p.d ? pb[(long long)(k0 + k + e) * (2 + kMaxD) + 2 + c] : 0.f;
#pragma unroll
      for (int e = 0; e < kAhead; ++e) {
        if (k + e >= n) break;
        L = fmaf(w[k + e], lw[k + e], L);
        Z = fmaf(w[k + e], zk[e], Z);
      }
    }
  }
  if (used == 0) __syncthreads();  // self is in (above: the weights' barrier)
  if (c < p.d)
    epilogue<TI>(p, bh, len, self, M, L, Z, c, vi,
                 reinterpret_cast<TI*>(p.out) + (long long)b * p.qsB + (long long)h * p.qsH);
}

template <typename TI, int NQ>
cudaError_t launch_t(const DecodeProblem& p, float* part, int n_chunks, cudaStream_t s) {
  int dev = 0, nsm = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) {
    note_failure("decode: device attributes");
    return e;
  }
  const long long heads = (long long)p.B * p.H;
  const bool qal = (reinterpret_cast<uintptr_t>(p.q) & 15u) == 0 &&
                   (p.qsB * (long long)sizeof(TI)) % 16 == 0 &&
                   (p.qsH * (long long)sizeof(TI)) % 16 == 0;
  constexpr int smem = Scan<TI, NQ>::kRing;
  auto allow = [&](const void* f) {
    const cudaError_t r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (r != cudaSuccess) note_failure("decode: shared memory");
    return r;
  };
  // One launch while its CTAs are all resident at once (two per SM fit) and a CTA has no more than
  // half of a partial CTA's rows; or as many, where the two passes would scan them by the same tiles
  // (below), or the cache is small (12K elements of K for every row of a chunk).  us, cluster against
  // partial and combine pass, caches that together exceed L2 / one cache that stays in it, bf16:
  // 12 heads, T 2048, d 64 8.6 against 16.5 / 8.2 against 9.7; 32 heads, T 2048, d 128 15.3 against
  // 19.3 / 14.3 against 11.9; 24 heads, T 4096, d 64 14.2 against 17.9 / 13.5 against 11.7; 38 heads,
  // T 4096, d 80 21.7 against 23.0 / 20.5 against 21.9.  Past the lines (32 heads, T 4096, d 128:
  // 24.3 against 22.6 / 23.2 against 15.2; T 8192, 12 heads: 18 against 16; 64 heads, T 1024, d 128:
  // 21 against 17) the CTAs are too few or come in waves.
  const bool steps = (p.d == 128 || p.d == 64) && qal;  // the partial pass in two steps
  if (kCluster * heads <= 2 * nsm &&
      (n_chunks <= kCluster / 2 ||
       (NQ > 0 && n_chunks <= kCluster &&
        (!steps || n_chunks * heads * p.d <= 12 * 1024)))) {
    if ((e = allow((const void*)cluster_kernel<TI, NQ>)) != cudaSuccess) return e;
    e = launch_pdl(cluster_kernel<TI, NQ>, dim3((unsigned)heads * kCluster), 32 * kClWarps, smem, s,
                   kCluster, p);
    if (e != cudaSuccess) note_failure("decode: cluster launch");
    return e;
  }
  const dim3 grid((unsigned)heads, (unsigned)n_chunks);
  if (NQ > 0 && steps && p.d == 128) {
    e = launch_pdl(partial_kernel<TI, 128>, grid, 32 * kWarps, 0, s, 1, p, part);
  } else if (NQ > 0 && steps) {
    e = launch_pdl(partial_kernel<TI, 64>, grid, 32 * kWarps, 0, s, 1, p, part);
  } else if constexpr (NQ > 0) {
    if ((e = allow((const void*)scan_kernel<TI, NQ>)) != cudaSuccess) return e;
    e = launch_pdl(scan_kernel<TI, NQ>, grid, 32 * kClWarps, smem, s, 1, p, part);
  } else {
    e = launch_pdl(partial_kernel<TI, 0>, grid, 32 * kWarps, 0, s, 1, p, part);
  }
  if (e != cudaSuccess) { note_failure("decode: partial pass launch"); return e; }
  e = launch_pdl(combine_kernel<TI>, dim3((unsigned)heads), kMaxD, 0, s, 1, p, (const float*)part,
                 n_chunks);
  if (e != cudaSuccess) note_failure("decode: combine launch");
  return e;
}

template <typename TI>
cudaError_t launch_d(const DecodeProblem& p, float* part, int n_chunks, cudaStream_t s) {
  // 16-byte row groups need aligned rows and a whole number of groups per row
  const bool vec = (reinterpret_cast<uintptr_t>(p.k) & 15u) == 0 &&
                   (reinterpret_cast<uintptr_t>(p.v) & 15u) == 0 &&
                   (p.sB * (long long)sizeof(TI)) % 16 == 0 &&
                   (p.sT * (long long)sizeof(TI)) % 16 == 0 &&
                   (p.sH * (long long)sizeof(TI)) % 16 == 0 && p.d % Vec<TI>::N == 0;
  constexpr int kQ = kMaxD / Vec<TI>::N / 4;
  if (!vec) return launch_t<TI, 0>(p, part, n_chunks, s);
  if (p.d <= kMaxD / 2) return launch_t<TI, kQ / 2>(p, part, n_chunks, s);
  return launch_t<TI, kQ>(p, part, n_chunks, s);
}

}  // namespace decode

int decode_chunks(int t_max) { return t_max > 1 ? (t_max - 1 + decode::kChunk - 1) / decode::kChunk : 1; }

size_t decode_workspace_bytes(int B, int H, int t_max) {
  return (size_t)B * H * decode_chunks(t_max) * (2 + decode::kMaxD) * sizeof(float);
}

cudaError_t launch_decode(const DecodeProblem& p, void* workspace, cudaStream_t s) {
  float* part = static_cast<float*>(workspace);
  const int n = decode_chunks(p.T);
  if (p.dtype == RELATION_F32) return decode::launch_d<float>(p, part, n, s);
  return decode::launch_d<__nv_bfloat16>(p, part, n, s);
}

}  // namespace rel
