// Warp-level building blocks of the fp32-compute path's tile kernels: bf16
// operand pieces in shared memory, ldmatrix fragment loads for both storage
// orders, m16n8k16 MMAs over the pieces, and 16-byte asynchronous copies.
#pragma once
#include "common.cuh"

namespace slim {
namespace simt {

typedef __nv_bfloat16 bf16;

// x = h + m + l with bf16 pieces: h = bf16(x), m = bf16(x - h), l = bf16(x - h - m)
// (each difference is exact in fp32), 24 bits of x in NP = 3 pieces, 16 in 2.
template <int NP>
__device__ __forceinline__ void split_bf16(float x, float (&pc)[NP]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    pc[i] = __bfloat162float(__float2bfloat16_rn(x));
    x = __fsub_rn(x, pc[i]);
  }
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float2 unpack2(uint32_t w) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w));
}
// the pieces of a pair of values as packed words
template <int NP>
__device__ __forceinline__ void split_pair(float x, float y, uint32_t (&w)[NP]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    w[i] = pack2(x, y);
    if (i + 1 < NP) {
      const float2 v = unpack2(w[i]);
      x = __fsub_rn(x, v.x);
      y = __fsub_rn(y, v.y);
    }
  }
}

// D += A B for one m16n8k16 tile: A 16 x 16 bf16 (row-major fragment), B
// 16 x 8 bf16 (column fragment), D fp32; one warp.
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Two n8 blocks: D0 | D1 += A B over the operands' pieces, products (i, j)
// with i + j < max(NA, NB), smallest first (b[j] = block 0's two registers,
// then block 1's).
template <int NA, int NB>
__device__ __forceinline__ void mma_pieces(float (&d0)[4], float (&d1)[4],
                                           const uint32_t (&a)[NA][4], const uint32_t (&b)[NB][4]) {
  constexpr int P = NA > NB ? NA : NB;
#pragma unroll
  for (int o = P - 1; o >= 0; --o)
#pragma unroll
    for (int i = 0; i <= o; ++i)
      if (i < NA && o - i < NB) {
        mma16816(d0, a[i], b[o - i][0], b[o - i][1]);
        mma16816(d1, a[i], b[o - i][2], b[o - i][3]);
      }
}

// The same into running sums that several k16 steps add to, in the backward: fp32
// problems (3 pieces) take each step's products from zero and add them in
// round-to-nearest, because an MMA's accumulation truncates (measured, d = 32
// fp32: dk 1.8e-6 from the exact value without, 8e-7 with it).
template <int NA, int NB>
__device__ __forceinline__ void mma_sum(float (&d0)[4], float (&d1)[4], const uint32_t (&a)[NA][4],
                                        const uint32_t (&b)[NB][4]) {
  if (NA < 3 && NB < 3) {
    mma_pieces<NA, NB>(d0, d1, a, b);
    return;
  }
  float t0[4] = {}, t1[4] = {};
  mma_pieces<NA, NB>(t0, t1, a, b);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    d0[c] += t0[c];
    d1[c] += t1[c];
  }
}

// One k16 step of a projection x . omega, whose error goes into an exponential:
// the leading pieces' product gets an accumulator of its own per step, added in
// round-to-nearest (an MMA's accumulation truncates, which would shrink a running
// sum step by step), and the small products accumulate apart in l0 | l1.
template <int NA, int NB>
__device__ __forceinline__ void mma_project(float (&d0)[4], float (&d1)[4], float (&l0)[4],
                                            float (&l1)[4], const uint32_t (&a)[NA][4],
                                            const uint32_t (&b)[NB][4]) {
  constexpr int P = NA > NB ? NA : NB;
#pragma unroll
  for (int o = P - 1; o >= 1; --o)
#pragma unroll
    for (int i = 0; i <= o; ++i)
      if (i < NA && o - i < NB) {
        mma16816(l0, a[i], b[o - i][0], b[o - i][1]);
        mma16816(l1, a[i], b[o - i][2], b[o - i][3]);
      }
  float h0[4] = {}, h1[4] = {};
  mma16816(h0, a[0], b[0][0], b[0][1]);
  mma16816(h1, a[0], b[0][2], b[0][3]);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    d0[c] += h0[c];
    d1[c] += h1[c];
  }
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p))
               : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const bf16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p))
               : "memory");
}
// Fragments of NP pieces (piece stride ps elements, row pitch elements).  The
// pitch is the row length plus 8 elements: the 8 rows an ldmatrix phase reads
// then start in 8 different 16-byte bank groups for every row length used.
//   ld_a:  A[r0..+15][k0..+15] stored [row][k]
//   ld_at: the same A stored [k][row]
//   ld_b:  B[k0..+15][n0..+15] stored [n][k]
//   ld_bt: the same B stored [k][n]
template <int NP>
__device__ __forceinline__ void ld_a(uint32_t (&a)[NP][4], const bf16* p, int ps, int pitch, int r0,
                                     int k0) {
  const int l = threadIdx.x & 31;
  p += (r0 + (l & 15)) * pitch + k0 + (l >> 4) * 8;
#pragma unroll
  for (int i = 0; i < NP; ++i) ldsm4(a[i], p + i * ps);
}
template <int NP>
__device__ __forceinline__ void ld_at(uint32_t (&a)[NP][4], const bf16* p, int ps, int pitch, int r0,
                                      int k0) {
  const int l = threadIdx.x & 31;
  p += (k0 + (l & 7) + (l >> 4) * 8) * pitch + r0 + ((l >> 3) & 1) * 8;
#pragma unroll
  for (int i = 0; i < NP; ++i) ldsm4t(a[i], p + i * ps);
}
template <int NP>
__device__ __forceinline__ void ld_b(uint32_t (&b)[NP][4], const bf16* p, int ps, int pitch, int n0,
                                     int k0) {
  const int l = threadIdx.x & 31;
  p += (n0 + (l & 7) + (l >> 4) * 8) * pitch + k0 + ((l >> 3) & 1) * 8;
#pragma unroll
  for (int i = 0; i < NP; ++i) ldsm4(b[i], p + i * ps);
}
template <int NP>
__device__ __forceinline__ void ld_bt(uint32_t (&b)[NP][4], const bf16* p, int ps, int pitch,
                                      int n0, int k0) {
  const int l = threadIdx.x & 31;
  p += (k0 + (l & 15)) * pitch + n0 + (l >> 4) * 8;
#pragma unroll
  for (int i = 0; i < NP; ++i) ldsm4t(b[i], p + i * ps);
}
// A fragment (16 rows x 16 k) from two n8 blocks of a product's accumulators:
// the accumulator layout of columns 2t, 2t + 1 is the fragment layout of k.
template <int NP>
__device__ __forceinline__ void acc_to_a(uint32_t (&a)[NP][4], const float (&c0)[4],
                                         const float (&c1)[4]) {
  uint32_t w[NP];
  split_pair<NP>(c0[0], c0[1], w);
#pragma unroll
  for (int i = 0; i < NP; ++i) a[i][0] = w[i];
  split_pair<NP>(c0[2], c0[3], w);
#pragma unroll
  for (int i = 0; i < NP; ++i) a[i][1] = w[i];
  split_pair<NP>(c1[0], c1[1], w);
#pragma unroll
  for (int i = 0; i < NP; ++i) a[i][2] = w[i];
  split_pair<NP>(c1[2], c1[3], w);
#pragma unroll
  for (int i = 0; i < NP; ++i) a[i][3] = w[i];
}

__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

__device__ __forceinline__ void cp16(bf16* dst, const bf16* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Programmatic dependent launches: wait for the work before this kernel in the
// stream, and let the next kernel's CTAs be scheduled as this one's drain.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

}  // namespace simt
}  // namespace slim
