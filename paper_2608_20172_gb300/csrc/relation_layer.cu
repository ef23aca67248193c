// relation_layer.cu -- the layer's transforms around the operator (Sec. 3.1-3.2,
// Eq. givens-rotation, App. A.2.2, App. B.3), as a producer pass in front of the
// Relation kernels and its gradient pass behind them.
//
//   RoPE (full head, RoFormer's interleaved pairs): pair c of the row at position m
//   (zero-based within its sequence) turns by m * base^(-2c/d):
//       (x_2c, x_2c+1) -> (x_2c cos - x_2c+1 sin, x_2c sin + x_2c+1 cos)
//   applied to P1 -> Q and P2 -> K; the information states are not rotated.
//   Givens mixing of head pairs (a, b) with angle theta_k, on every channel:
//       I~_a = cos I_a - sin I_b,   I~_b = sin I_a + cos I_b   (V = I~)
//   pairing A: (0,1), (2,3), ...; pairing B: (1,2), (3,4), ..., (H-1,0).
//   Gradients: the transposed rotations, and
//       dtheta_k = sum dI~_a (-sin I_a - cos I_b) + dI~_b (cos I_a - sin I_b).
//
// Both passes are HBM-bound (prep reads P1, P2, I and writes Q, K, V; grad reads dQ, dK,
// dV, I and writes dP1, dP2, dI): CTAs of 8 or 16 positions of a sequence move 8-element
// vectors (16 bytes in bf16).  The rotation angles of the CTA's positions are tabulated
// once in shared memory and reused by every head: m * base^(-2c/d) is formed and reduced
// modulo 2 pi as a sum of two floats (positions reach 16k, where an fp32 angle would be off
// by ~1e-3 rad; past 32k in fp64) from frequencies that come with the launch, then its cosine and
// sine are taken in fp32.  (In fp64, with an fp64 log and exp per CTA, this chip's fp64 pipe bounded
// both passes; the rotations and the mixing are CTAs of their own, so that the tables hide.
// B 4, H 8, T 4096, d 80: prep 48 -> 26 us, grad 63 -> 36; B 2, H 16, T 16384, d 128: 159 ->
// 122 us (6.6 TB/s), 196 -> 149 (6.3).)  dtheta is summed per CTA in a fixed
// order and the partials are added up in fp64 by a second kernel, one block per head
// pair (deterministic).
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace rel {
namespace layer {

// Positions and threads of a CTA.  prep: small CTAs, whose last wave is short (16 and 256 take
// 28.4 instead of 25.5 us at B 4, H 8, T 4096, d 80, 29.9 instead of 27.4 at B 32, T 1024, d 48).
// grad keeps 16, whose dtheta partials its workspace holds.
constexpr int kPrepTok = 8, kPrepThreads = 128;
constexpr int kTok = 16, kThreads = 256;
constexpr int kMaxD = 256;     // head size limit of these passes
constexpr int kMaxPairs = 128; // H / 2 limit

template <typename TI>
struct Vec8;
template <>
struct Vec8<__nv_bfloat16> {
  using Raw = uint4;
  __device__ static Raw load(const __nv_bfloat16* p) { return *reinterpret_cast<const uint4*>(p); }
  __device__ static void unpack(const Raw& w, float (&x)[8]) {
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u[i]));
      x[2 * i] = f.x;
      x[2 * i + 1] = f.y;
    }
  }
  __device__ static void store(void* p, const float (&x)[8]) {
    *reinterpret_cast<uint4*>(p) = make_uint4(pack_bf16x2(x[0], x[1]), pack_bf16x2(x[2], x[3]),
                                              pack_bf16x2(x[4], x[5]), pack_bf16x2(x[6], x[7]));
  }
};
template <>
struct Vec8<float> {
  struct Raw {
    float4 a, b;
  };
  __device__ static Raw load(const float* p) {
    return {reinterpret_cast<const float4*>(p)[0], reinterpret_cast<const float4*>(p)[1]};
  }
  __device__ static void unpack(const Raw& w, float (&x)[8]) {
    x[0] = w.a.x; x[1] = w.a.y; x[2] = w.a.z; x[3] = w.a.w;
    x[4] = w.b.x; x[5] = w.b.y; x[6] = w.b.z; x[7] = w.b.w;
  }
  __device__ static void store(void* p, const float (&x)[8]) {
    reinterpret_cast<float4*>(p)[0] = make_float4(x[0], x[1], x[2], x[3]);
    reinterpret_cast<float4*>(p)[1] = make_float4(x[4], x[5], x[6], x[7]);
  }
};

template <int TOK>
struct Tables {
  float cs[TOK][kMaxD / 2], sn[TOK][kMaxD / 2];  // RoPE of the CTA's positions
};

// The kernels' parameters: the problem and the frequencies base^(-2c/d), each as a sum of two
// floats (48 bits).
struct Args {
  LayerProblem p;
  float w_hi[kMaxD / 2], w_lo[kMaxD / 2];
};

// Positions whose angles come from turn: up to there they are as exact as fp64's, both being
// rounded to fp32 in the end (against 64 bits over d 48 to 256, bases 1 to 5e5: rms 4.66e-8 rad with
// either, at most 1.193e-7 against 1.192e-7 below 2^15 positions; 1.20e-7 at 2^17, 1.49e-7 at 2^22).
constexpr int kTurnPositions = 1 << 15;

// m * w modulo 2 pi (|r| <= pi + rounding) for a position m and w = w_hi + w_lo <= 1: the product
// and n 2 pi are kept as rounded value and exact remainder (two-product by fma; their leading
// parts are close, so that their difference is exact), 2 pi as a sum of two floats (48 bits).
// The _rn forms: a product that was contracted into the difference would have its remainder
// counted twice.
__device__ __forceinline__ float turn(float m, float w_hi, float w_lo) {
  constexpr float kTwoPiHi = 6.28318530717958647692f;
  constexpr float kTwoPiLo = (float)(6.28318530717958647692 - (double)kTwoPiHi);
  const float a = __fmul_rn(m, w_hi);
  const float a_lo = fmaf(m, w_lo, fmaf(m, w_hi, -a));
  const float n = rintf(__fmul_rn(a, 0.15915494309189533577f));
  const float q = __fmul_rn(n, kTwoPiHi);
  const float q_lo = fmaf(n, kTwoPiLo, fmaf(n, kTwoPiHi, -q));
  return __fadd_rn(__fsub_rn(a, q), __fsub_rn(a_lo, q_lo));
}

// cos / sin of m * base^(-2c/d) for the CTA's positions
template <int TOK, int NT>
__device__ __forceinline__ void fill_tables(Tables<TOK>& tb, const Args& ar, int t0) {
  const LayerProblem& p = ar.p;
  const int half = p.d / 2;
  for (int e = threadIdx.x; e < TOK * half; e += NT) {
    const int tt = e / half, c = e % half;
    float r;
    if (t0 < kTurnPositions && p.rope_base >= 1.0f) {
      r = turn((float)(t0 + tt), ar.w_hi[c], ar.w_lo[c]);
    } else {  // positions or frequencies past turn's range: fp64
      const double a = (double)(t0 + tt) * exp(-2.0 * (double)c / (double)p.d * log((double)p.rope_base));
      r = (float)fma(-rint(a * 0.15915494309189533576888376337251),
                     6.283185307179586476925286766559, a);
    }
    float s, co;
    sincosf(r, &s, &co);
    tb.cs[tt][c] = co;
    tb.sn[tt][c] = s;
  }
}

// heads of Givens pair k
__device__ __forceinline__ void pair_heads(const LayerProblem& p, int k, int& a, int& b) {
  a = p.pairing == 0 ? 2 * k : 2 * k + 1;
  b = p.pairing == 0 ? 2 * k + 1 : (2 * k + 2) % p.H;
}

// rotate the 4 pairs of an 8-element chunk starting at channel 8 u by +-angle
template <int TOK>
__device__ __forceinline__ void rotate8(float (&x)[8], const Tables<TOK>& tb, int tt, int u,
                                        float sgn) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float co = tb.cs[tt][4 * u + i], s = sgn * tb.sn[tt][4 * u + i];
    const float x0 = x[2 * i], x1 = x[2 * i + 1];
    x[2 * i] = x0 * co - x1 * s;
    x[2 * i + 1] = x0 * s + x1 * co;
  }
}

// A CTA's sequence and positions.  Even CTAs rotate, odd ones mix: a rotating CTA's first
// loads are in flight while it tabulates the angles, and the mixing CTAs beside it have none
// to wait for.
struct Where {
  int b, t0, nt;
};
template <int TOK>
__device__ __forceinline__ Where where(const LayerProblem& p) {
  const int n_tt = (p.T + TOK - 1) / TOK, w = (int)(blockIdx.x >> 1);
  const int t0 = (w % n_tt) * TOK;
  return {w / n_tt, t0, min(TOK, p.T - t0)};
}

// RoPE (sgn = +1) or its transpose (sgn = -1) of in1 -> out1 and in2 -> out2 over the
// CTA's (position, head, chunk) items, two items per thread and iteration so that four
// 16-byte loads are in flight (the first ones during the tables).
template <typename TI, int TOK, int NT>
__device__ __forceinline__ void rope_pass(Tables<TOK>& tb, const Args& ar, const Where& at, float sgn) {
  using V = Vec8<TI>;
  const LayerProblem& p = ar.p;
  const int nu = p.d / 8;
  const int n = at.nt * p.H * nu;
  const long long base = (long long)at.b * p.sB;
  const TI* in1 = reinterpret_cast<const TI*>(p.in1);
  const TI* in2 = reinterpret_cast<const TI*>(p.in2);
  struct Item {
    long long off;
    int tt, u;
  };
  auto item = [&](int e) {  // (clamped: a thread past the end reloads the last item)
    e = min(e, n - 1);
    const int r = e / nu, h = r % p.H, tt = r / p.H;
    Item i;
    i.u = e - r * nu;
    i.tt = tt;
    i.off = base + (long long)(at.t0 + tt) * p.sT + (long long)h * p.sH + 8 * i.u;
    return i;
  };
  auto put = [&](const Item& i, const typename V::Raw& a, const typename V::Raw& b) {
    float x[8], y[8];
    V::unpack(a, x);
    V::unpack(b, y);
    rotate8(x, tb, i.tt, i.u, sgn);
    rotate8(y, tb, i.tt, i.u, sgn);
    V::store(reinterpret_cast<TI*>(p.out1) + i.off, x);
    V::store(reinterpret_cast<TI*>(p.out2) + i.off, y);
  };
  Item i0 = item(threadIdx.x), i1 = item(threadIdx.x + NT);
  typename V::Raw x0 = V::load(in1 + i0.off), y0 = V::load(in2 + i0.off);
  typename V::Raw x1 = V::load(in1 + i1.off), y1 = V::load(in2 + i1.off);
  fill_tables<TOK, NT>(tb, ar, at.t0);
  __syncthreads();
  for (int e = threadIdx.x; e < n; e += 2 * NT) {
    if (e != (int)threadIdx.x) {
      i0 = item(e);
      i1 = item(e + NT);
      x0 = V::load(in1 + i0.off);
      y0 = V::load(in2 + i0.off);
      x1 = V::load(in1 + i1.off);
      y1 = V::load(in2 + i1.off);
    }
    put(i0, x0, y0);
    if (e + NT < n) put(i1, x1, y1);
  }
}

template <typename TI>
__global__ void __launch_bounds__(kPrepThreads) prep_kernel(const __grid_constant__ Args ar) {
  using V = Vec8<TI>;
  const LayerProblem& p = ar.p;
  const Where at = where<kPrepTok>(p);
  pdl_wait_and_launch();
  if (!(blockIdx.x & 1)) {  // Q = RoPE(P1), K = RoPE(P2)
    __shared__ Tables<kPrepTok> tb;
    rope_pass<TI, kPrepTok, kPrepThreads>(tb, ar, at, 1.f);
    return;
  }
  // Givens mixing of the information states: (token, pair, chunk) items, two per thread and
  // iteration
  const int nu = p.d / 8, np = p.H / 2, n = at.nt * np * nu;
  const long long base = (long long)at.b * p.sB;
  const TI* in = reinterpret_cast<const TI*>(p.in3);
  TI* out = reinterpret_cast<TI*>(p.out3);
  for (int e0 = threadIdx.x; e0 < n; e0 += 2 * kPrepThreads) {
    typename V::Raw ra[2], rb[2];
    long long oa[2], ob[2];
    float th[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int e = min(e0 + i * kPrepThreads, n - 1);
      const int r = e / nu, k = r % np, tt = r / np;
      int ha, hb;
      pair_heads(p, k, ha, hb);
      const long long row = base + (long long)(at.t0 + tt) * p.sT + 8 * (e - r * nu);
      oa[i] = row + (long long)ha * p.sH;
      ob[i] = row + (long long)hb * p.sH;
      ra[i] = V::load(in + oa[i]);
      rb[i] = V::load(in + ob[i]);
      th[i] = p.theta[k];
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (e0 + i * kPrepThreads >= n) break;
      float ia[8], ib[8], va[8], vb[8], s, co;
      sincosf(th[i], &s, &co);
      V::unpack(ra[i], ia);
      V::unpack(rb[i], ib);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        va[j] = co * ia[j] - s * ib[j];
        vb[j] = s * ia[j] + co * ib[j];
      }
      V::store(out + oa[i], va);
      V::store(out + ob[i], vb);
    }
  }
}

template <typename TI>
__global__ void __launch_bounds__(kThreads) grad_kernel(const __grid_constant__ Args ar) {
  using V = Vec8<TI>;
  const LayerProblem& p = ar.p;
  const Where at = where<kTok>(p);
  pdl_wait_and_launch();
  if (!(blockIdx.x & 1)) {  // transposed RoPE: dP1 from dQ, dP2 from dK
    __shared__ Tables<kTok> tb;
    rope_pass<TI, kTok, kThreads>(tb, ar, at, -1.f);
    return;
  }
  __shared__ float part[kThreads / 32][kMaxPairs], tc[kMaxPairs], ts[kMaxPairs];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int k = threadIdx.x; k < p.H / 2; k += kThreads) {
    float s, co;
    sincosf(p.theta[k], &s, &co);
    tc[k] = co;
    ts[k] = s;
  }
  for (int k = lane; k < p.H / 2; k += 32) part[warp][k] = 0.f;
  __syncthreads();
  const int nu = p.d / 8, t0 = at.t0;
  const long long base = (long long)at.b * p.sB;
  // transposed Givens: dI from dV = dI~, and dtheta.  The loop runs the same number of
  // times on every lane (items past the end are idle), so the warp can reduce dtheta
  // over runs of lanes with the same pair (items are ordered chunk, pair, position) and
  // add each run's sum to its pair's slot in lane order (deterministic).
  const int np = p.H / 2;
  const int n_items = at.nt * np * nu;
  for (int e0 = 0; e0 < n_items; e0 += kThreads) {
    const int e = e0 + (int)threadIdx.x;
    const bool live = e < n_items;
    const int ec = live ? e : 0;
    const int rr = ec / nu, u = ec - rr * nu, k = rr % np, tt = rr / np;
    float dt = 0.f;
    if (live) {
      int ha, hb;
      pair_heads(p, k, ha, hb);
      const long long row = base + (long long)(t0 + tt) * p.sT + 8 * u;
      const long long oa = row + (long long)ha * p.sH, ob = row + (long long)hb * p.sH;
      float ga[8], gb[8], ia[8], ib[8], da[8], db[8];
      const typename V::Raw r1 = V::load(reinterpret_cast<const TI*>(p.in3) + oa);
      const typename V::Raw r2 = V::load(reinterpret_cast<const TI*>(p.in3) + ob);
      const typename V::Raw r3 = V::load(reinterpret_cast<const TI*>(p.in4) + oa);
      const typename V::Raw r4 = V::load(reinterpret_cast<const TI*>(p.in4) + ob);
      V::unpack(r1, ga);
      V::unpack(r2, gb);
      V::unpack(r3, ia);
      V::unpack(r4, ib);
      const float co = tc[k], s = ts[k];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        da[i] = co * ga[i] + s * gb[i];
        db[i] = -s * ga[i] + co * gb[i];
        dt += ga[i] * (-s * ia[i] - co * ib[i]) + gb[i] * (co * ia[i] - s * ib[i]);
      }
      Vec8<TI>::store(reinterpret_cast<TI*>(p.out3) + oa, da);
      Vec8<TI>::store(reinterpret_cast<TI*>(p.out3) + ob, db);
    }
    // runs of consecutive lanes with the same pair (idle lanes form runs of their own)
    const int key = live ? k : -1 - lane;
    const int kprev = __shfl_up_sync(0xffffffffu, key, 1);
    const bool head = lane == 0 || kprev != key;
    const unsigned heads = __ballot_sync(0xffffffffu, head);
    const int first = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));  // my run's first lane
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float t = __shfl_up_sync(0xffffffffu, dt, o);
      if (lane - o >= first) dt += t;
    }
    const int knext = __shfl_down_sync(0xffffffffu, key, 1);
    const bool tail = lane == 31 || knext != key;
    const int run = __popc(heads & (0xffffffffu >> (31 - lane))) - 1;
    const int n_runs = __popc(heads);
    for (int r = 0; r < n_runs; ++r) {
      if (tail && live && run == r) part[warp][k] += dt;
      __syncwarp();
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < np; k += kThreads) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) s += part[w][k];
    p.dtheta_part[(long long)(blockIdx.x >> 1) * np + k] = s;
  }
}

// dtheta_k = sum over CTAs of the partials, in fp64 and a fixed order; one block per pair
__global__ void __launch_bounds__(256) dtheta_kernel(LayerProblem p, int n_cta) {
  __shared__ double red[8];
  const int np = p.H / 2, k = blockIdx.x;
  pdl_wait_and_launch();
  double s = 0.0;
  for (int c = threadIdx.x; c < n_cta; c += 256) s += (double)p.dtheta_part[(long long)c * np + k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) s += red[w];
    p.dtheta[k] = (float)s;
  }
}

Args args_of(const LayerProblem& p) {
  Args ar;
  ar.p = p;
  const double lnb = log((double)p.rope_base);
  for (int c = 0; c < p.d / 2; ++c) {
    const double w = exp(-2.0 * (double)c / (double)p.d * lnb);
    ar.w_hi[c] = (float)w;
    ar.w_lo[c] = (float)(w - (double)ar.w_hi[c]);
  }
  return ar;
}

int per_sequence(const LayerProblem& p, int tok) { return p.T / tok + (p.T % tok != 0); }

// A grid holds 2^31 - 1 CTAs, two for every `tok` positions of a sequence: more sequences than that
// come in several launches.
template <typename K>
cudaError_t launch_sequences(K kernel, const LayerProblem& p, int tok, unsigned threads, cudaStream_t s) {
  Args ar = args_of(p);
  const int per = per_sequence(p, tok), most = 0x7fffffff / (2 * per);
  const long long esz = p.dtype == RELATION_F32 ? 4 : 2;
  for (long long b = 0; b < p.B; b += most) {
    const int n = (int)(p.B - b < most ? p.B - b : most);
    const long long off = b * p.sB * esz;
    auto in = [&](const void* x) -> const void* { return x ? static_cast<const char*>(x) + off : x; };
    auto out = [&](void* x) -> void* { return x ? static_cast<char*>(x) + off : x; };
    ar.p.B = n;
    ar.p.in1 = in(p.in1); ar.p.in2 = in(p.in2); ar.p.in3 = in(p.in3); ar.p.in4 = in(p.in4);
    ar.p.out1 = out(p.out1); ar.p.out2 = out(p.out2); ar.p.out3 = out(p.out3);
    if (p.dtheta_part) ar.p.dtheta_part = p.dtheta_part + b * per * (p.H / 2);
    const cudaError_t e = launch_pdl(kernel, dim3(2u * n * per), threads, 0, s, 1, ar);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace layer

bool layer_supports(relation_dtype dt, int d, int H) {
  return (dt == RELATION_F32 || dt == RELATION_BF16) && d >= 8 && d % 8 == 0 &&
         d <= layer::kMaxD && H >= 2 && H % 2 == 0 && H / 2 <= layer::kMaxPairs;
}

size_t layer_grad_workspace_bytes(int B, int T, int H) {
  return (size_t)B * ((T + layer::kTok - 1) / layer::kTok) * (H / 2) * sizeof(float);
}

cudaError_t launch_layer_prep(const LayerProblem& p, cudaStream_t s) {
  const cudaError_t e = layer::launch_sequences(
      p.dtype == RELATION_F32 ? layer::prep_kernel<float> : layer::prep_kernel<__nv_bfloat16>, p,
      layer::kPrepTok, layer::kPrepThreads, s);
  if (e != cudaSuccess) note_failure("layer prep: launch");
  return e;
}

cudaError_t launch_layer_grad(const LayerProblem& p, cudaStream_t s) {
  cudaError_t e = layer::launch_sequences(
      p.dtype == RELATION_F32 ? layer::grad_kernel<float> : layer::grad_kernel<__nv_bfloat16>, p,
      layer::kTok, layer::kThreads, s);
  if (e != cudaSuccess) { note_failure("layer grad: launch"); return e; }
  e = launch_pdl(layer::dtheta_kernel, dim3(p.H / 2), 256, 0, s, 1, p,
                 p.B * layer::per_sequence(p, layer::kTok));
  if (e != cudaSuccess) note_failure("layer grad: dtheta launch");
  return e;
}

}  // namespace rel
