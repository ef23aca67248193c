// relation_linear_tc.cuh -- shared pieces of the chunked tensor-core Linear Relation
// kernels (relation_linear_tc.cu: forward, state scans; relation_linear_tc_bwd.cu:
// backward): block size, the workspace view, shared-memory layout helpers, tensor maps.
#pragma once

#include <cudaTypedefs.h>
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace rel {
namespace tc {
bool make_tmap_bf16(CUtensorMap* m, const void* base, const Problem& p, int rows);
}
namespace lintc {


constexpr int LT = 128;          // tokens per block
constexpr int NC = 64;           // information columns per CTA
constexpr float kClampLog2 = 120.0f;

// Modes of the kernel: SEQ walks all blocks of a (head, split) in order with the state in
// TMEM; the chunk-parallel pair takes any block by itself: DELTA writes the block's state
// contribution sum_j KL_j I~_j^T and decay a_L (fp32) to the workspace, OUT reads the
// state the block starts from (bf16, produced by scan_kernel) and writes the block's Y.
// BOTH (the backward, d_h = 64) is DELTA together with the block's contribution to the
// state's adjoint, Qs^T dY.
enum : int { MODE_SEQ = 0, MODE_DELTA = 1, MODE_OUT = 2, MODE_BOTH = 3 };

// Workspace of the chunk-parallel forms, per (head, split, block): dC [D][64] fp32 (after the
// scan every row's first 128 bytes hold the row of the state entering the block, bf16), the
// decay g [D] fp32 and, for the backward, dQ [D][64] likewise (the adjoint leaving the block).
struct LinCp {
  float* dC;
  float* dQ;
  float* g;
  int nb;
};

// B_LOAD, B_FREE, B_EPI: one per input stage (stage s at + s)
enum : int { B_LOAD = 0, B_FREE = 2, B_EPI = 4, B_OPS = 6, B_C0, B_S, B_A, B_E, B_STATE, NBAR };
// the one-block modes have one stage: I~'s (and the state's) loads, and Y has left Qs
enum : int { B_LOADV = B_LOAD + 1, B_QFREE = B_FREE };

__device__ __forceinline__ void drain_wait(uint32_t bar, uint32_t parity) {
  const unsigned long long t0 = globaltimer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (globaltimer_ns() - t0 > 20ull * 1000ull * 1000ull) return;
  }
}
// 2-D tiled load into shared memory, completing on `bar` (transaction bytes).
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
template <int NG>
__device__ __forceinline__ void ew_sync() {  // the elementwise warpgroups
  asm volatile("bar.sync 1, %0;" ::"n"(NG * 128) : "memory");
}
// byte offset of element (row r, column c) in a tile of 128-byte-swizzled rows of 64
// bf16 columns, blocks of `rows` rows per 64 columns
__device__ __forceinline__ uint32_t swz(int r, int c, int rows) {
  return (uint32_t)((c >> 6) * rows * 128 + r * 128 + ((((c & 63) >> 3) ^ (r & 7)) << 4) +
                    (c & 7) * 2);
}
// log2 of a retention.  The flushing form takes one instruction where the other scales denormal
// arguments; those (and 0) give -150 instead: any factor that holds one is 0 in fp32 or beyond
// kClampLog2 with the true logarithm (below -126) as well.  NaN stays NaN.
__device__ __forceinline__ float log2_alpha(float a) {
  float x, y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(a));
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(x), "f"(-150.0f));
  return y;
}
// The same for one exponent already reported (NaN stays NaN)
__device__ __forceinline__ float clamp_exponent(float dm) {
  float y;
  asm("{\n\t.reg .f32 t;\n\tmax.NaN.f32 t, %1, %2;\n\tmin.NaN.f32 %0, t, %3;\n\t}"
      : "=f"(y)
      : "f"(dm), "f"(-kClampLog2), "f"(kClampLog2));
  return y;
}
// Exponents of intra-block factors clamped to +-kClampLog2 (the test for all first: none is, but
// for channels whose result is reported as not exact)
template <int N>
__device__ __forceinline__ void clamp_exponents(float (&dm)[N], bool& clamped) {
  float mx = 0.f;
#pragma unroll
  for (int i = 0; i < N; ++i) mx = fmaxf(mx, fabsf(dm[i]));
  if (mx > kClampLog2) {
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (fabsf(dm[i]) > kClampLog2) dm[i] = copysignf(kClampLog2, dm[i]);
    clamped = true;
  }
}
// Ask Self's sums of token t over its D channels (p1, p2: 128-byte-swizzled bf16 tiles),
// those of `which`: 1 p1 . p2, 2 |p1|^2, 4 |p2|^2.  Each is one chain of multiply-adds in
// channel order whichever thread takes it.  ALL = 7 where `which` is 7 at compile time.
template <int D, int ALL>
__device__ __forceinline__ void ask_self_sums(const uint8_t* p1s, const uint8_t* p2s, int t,
                                              int which, float* dot, float* n1, float* n2) {
  auto pass = [&](auto f, bool r1, bool r2) {
#pragma unroll
    for (int k = 0; k < D / 8; ++k) {
      const uint32_t off = (k >> 3) * LT * 128 + t * 128 + (((k & 7) ^ (t & 7)) << 4);
      uint4 a4 = make_uint4(0, 0, 0, 0), b4 = a4;
      if (r1) a4 = *reinterpret_cast<const uint4*>(p1s + off);
      if (r2) b4 = *reinterpret_cast<const uint4*>(p2s + off);
      const uint32_t aw[4] = {a4.x, a4.y, a4.z, a4.w}, bw[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        f(__bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&aw[e])),
          __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bw[e])));
    }
  };
  float s0 = 0.f, s1 = 0.f, s2 = 0.f;
  if (ALL == 7) {
    pass([&](float2 x, float2 y) {
      s0 = fmaf(x.x, y.x, fmaf(x.y, y.y, s0));
      s1 = fmaf(x.x, x.x, fmaf(x.y, x.y, s1));
      s2 = fmaf(y.x, y.x, fmaf(y.y, y.y, s2));
    }, true, true);
    dot[t] = s0;
    n1[t] = s1;
    n2[t] = s2;
  } else if (which == 1) {
    pass([&](float2 x, float2 y) { s0 = fmaf(x.x, y.x, fmaf(x.y, y.y, s0)); }, true, true);
    dot[t] = s0;
  } else if (which == 2) {
    pass([&](float2 x, float2) { s1 = fmaf(x.x, x.x, fmaf(x.y, x.y, s1)); }, true, false);
    n1[t] = s1;
  } else {
    pass([&](float2, float2 y) { s2 = fmaf(y.x, y.x, fmaf(y.y, y.y, s2)); }, false, true);
    n2[t] = s2;
  }
}
// element (token, channel) of [d / 32][128][32] fp32 tiles written by the swizzled
// retention map: the 16-byte groups of a token's 128-byte row permuted by (token & 7)
__device__ __forceinline__ int al_swz(int tok, int ch) {
  return (ch >> 5) * (LT * 32) + tok * 32 + ((((ch & 31) >> 2) ^ (tok & 7)) << 2) + (ch & 3);
}


// 4-D map over the [B][T][H][d] fp32 retention: boxes of 32 channels x 128 tokens, no
// swizzle, or (swz) with the 128-byte swizzle, so that a thread per token reading its row
// and a thread per channel reading a column both spread over the banks (al_swz).
inline bool make_tmap_alpha(CUtensorMap* m, const LinearProblem& p, bool swz = false) {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return false;
    fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  }
  cuuint64_t dims[4] = {(cuuint64_t)p.d, (cuuint64_t)p.T, (cuuint64_t)p.H, (cuuint64_t)p.B};
  cuuint64_t strides[3] = {(cuuint64_t)p.sT * 4, (cuuint64_t)p.sH * 4, (cuuint64_t)p.sB * 4};
  cuuint32_t box[4] = {32, (cuuint32_t)LT, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(p.alpha), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            swz ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D map over the bf16 state rows of the workspace: [rows][64] at a pitch of 256 bytes, boxes
// of D rows, 128-byte swizzle (the MN-major B layout of the E = Qs C_0 product).
inline bool make_tmap_c0(CUtensorMap* m, void* base, long long rows, int d) {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return false;
    fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  }
  cuuint64_t dims[2] = {64, (cuuint64_t)rows};
  cuuint64_t strides[1] = {256};
  cuuint32_t box[2] = {64, (cuuint32_t)d};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

size_t bwd_bytes(long long heads, long long nb, int d, LinCp* cp, void* base);
cudaError_t launch_states(const LinearProblem& lp, const void* dy, void* workspace, cudaStream_t s);

}  // namespace lintc
}  // namespace rel
