// Arithmetic shared by the fp32-compute path's kernels: operand pieces, features
// by FMA projections, and programmatic dependent launches.
#pragma once
#include <math.h>

#include "profiler.h"
#include "warp_mma.cuh"

namespace slim {
namespace simt {

constexpr int kThreads = 256;  // 8 warps
constexpr int kSmemMax = 232448;  // shared memory of a CTA
template <typename IO> struct Pieces;
template <> struct Pieces<bf16> { static constexpr int NX = 1, NS = 2; };
template <> struct Pieces<float> { static constexpr int NX = 3, NS = 3; };

__device__ __forceinline__ void load8(const bf16* p, float (&v)[8]) {
  const uint4 r = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = unpack2(w[i]);
    v[2 * i] = f.x;
    v[2 * i + 1] = f.y;
  }
}
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
// 8 consecutive values as NP pieces (piece stride ps)
template <int NP>
__device__ __forceinline__ void store_pieces8(bf16* dst, int ps, const float (&v)[8]) {
  uint32_t w[4][NP];
#pragma unroll
  for (int i = 0; i < 4; ++i) split_pair<NP>(v[2 * i], v[2 * i + 1], w[i]);
#pragma unroll
  for (int p = 0; p < NP; ++p)
    *reinterpret_cast<uint4*>(dst + p * ps) = make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
}

// a staged element's value (the sum of its pieces, exact for a caller's rows)
template <int NP>
__device__ __forceinline__ float staged(const bf16* p, int ps) {
  float v = __bfloat162float(p[(NP - 1) * ps]);
#pragma unroll
  for (int i = NP - 2; i >= 0; --i) v += __bfloat162float(p[i * ps]);
  return v;
}

// x . omega as a compensated dot product (FMA TwoProduct and TwoSum, about 48
// bits; Ogita, Rump and Oishi's Dot2): decides ReLU's branch where the
// projection's own error could.
static __device__ __noinline__ float dot2_staged(const float* x, const float* om, int stride, int d) {
  float sh = 0.f, sl = 0.f;
  for (int j = 0; j < d; ++j) {
    const float xw = x[j], ow = om[j * stride];
    const float p = __fmul_rn(xw, ow), ep = __fmaf_rn(xw, ow, -p);
    float t, e;
    two_sum(sh, p, t, e);
    sh = t;
    sl = __fadd_rn(sl, __fadd_rn(e, ep));
  }
  return __fadd_rn(sh, sl);
}
// g of one element from its FMA projection `dot`: norm2 = |x|^2, om_norm =
// |omega|, x and om (stride os) in shared memory for ReLU's recheck.
template <int D>
__device__ __forceinline__ float feature_fp(int feature, float dot, float norm2, float om_norm,
                                            float inv_sqrt_m, const float* x, const float* om, int os) {
  if (feature == SLIM_FEAT_EXP) return expf(dot - 0.5f * norm2) * inv_sqrt_m;
  // error bound of an fp32 dot product of length D, times a safety factor 2
  const float gamma = 2.f * (float)(D + 2) * 5.9604645e-08f;
  if (fabsf(dot) <= gamma * om_norm * sqrtf(norm2)) dot = dot2_staged(x, om, os, D);
  return dot > 0.f ? dot * inv_sqrt_m : 0.f;
}

// |x|^2 of one row of D floats in shared memory, by one warp: strided terms,
// then a butterfly
template <int D>
__device__ __forceinline__ float warp_norm2(const float* x) {
  float s = 0.f;
#pragma unroll
  for (int j = threadIdx.x % 32; j < D; j += 32) s = fmaf(x[j], x[j], s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// warp_norm2's sums, term for term, by one thread (16-byte aligned x)
template <int D>
__device__ __forceinline__ float thread_norm2(const float* x) {
  float s[32] = {};
#pragma unroll
  for (int j = 0; j < D; j += 4) {
    const float4 v = *reinterpret_cast<const float4*>(x + j);
    s[j % 32] = fmaf(v.x, v.x, s[j % 32]);
    s[j % 32 + 1] = fmaf(v.y, v.y, s[j % 32 + 1]);
    s[j % 32 + 2] = fmaf(v.z, v.z, s[j % 32 + 2]);
    s[j % 32 + 3] = fmaf(v.w, v.w, s[j % 32 + 3]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < o; ++i) s[i] += s[i + o];
  return s[0];
}

// the fp32 value of staged pieces, smallest piece first
template <int NP>
__device__ __forceinline__ void add_pieces8(const bf16* p, int ps, float (&v)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = 0.f;
#pragma unroll
  for (int q = NP - 1; q >= 0; --q) {
    float w[8];
    load8(p + q * ps, w);
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] += w[i];
  }
}
// the same of one element
template <int NP>
__device__ __forceinline__ float staged_sum(const bf16* p, int ps) {
  float v = 0.f;
#pragma unroll
  for (int q = NP - 1; q >= 0; --q) v += __bfloat162float(p[q * ps]);
  return v;
}
template <int NP>
__device__ __forceinline__ float round_pieces(float x) {
  float pc[NP];
  split_bf16<NP>(x, pc);
  float v = 0.f;
#pragma unroll
  for (int q = NP - 1; q >= 0; --q) v += pc[q];
  return v;
}
// D += A b for one n8 block, A's pieces smallest first
template <int NA>
__device__ __forceinline__ void mma_n8(float (&d)[4], const uint32_t (&a)[NA][4], uint32_t b0, uint32_t b1) {
#pragma unroll
  for (int i = NA - 1; i >= 0; --i) mma16816(d, a[i], b0, b1);
}
constexpr uint32_t kOnes = 0x3f803f80u;  // two bf16 ones

__device__ __forceinline__ void store2(bf16* p, float x, float y) {
  *reinterpret_cast<uint32_t*>(p) = pack2(x, y);
}
__device__ __forceinline__ void store2(float* p, float x, float y) {
  *reinterpret_cast<float2*>(p) = make_float2(x, y);
}

// A launch as a programmatic dependent of the kernel before it in the stream: its
// CTAs may start once every CTA of that kernel has called pdl_launch.  Every kernel
// of a launch sequence calls pdl_wait before pdl_launch, so when a kernel starts, all
// but the one directly ahead of it have completed: before its own pdl_wait it reads
// the caller's tensors and what older kernels left (never the kernel ahead's output),
// and writes shared memory only.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, unsigned block, size_t smem,
                       cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace simt
}  // namespace slim
