// Tile kernels of the fp32-compute path.
//
// A frame is 64 rows of one chain: one tile of 64 or 48 rows, or two or four tiles
// of short slices.  Operands are split once into bf16 pieces
// (NX for a caller's rows: 1 for bf16, 3 for fp32; NS for everything computed:
// 2 for bf16 problems, 3 for fp32 ones) when they enter shared memory or become
// an MMA fragment, and every product of a tile stays in the CTA: nothing but
// the tile's state, its g(K) and its results goes through global memory.
// Products run as warp MMAs (m16n8k16): the pieces of a 64-row tile with
// M = 256 features would leave no room for tcgen05's 128-row operand tiles, and
// an accumulator that already sits in registers becomes the next product's
// operand without a trip through shared memory.  m16n8k16 bf16 measured 600
// TFLOP/s on a GB300 (1.86 PFLOP/s for tcgen05), with 3 (bf16) or 6 (fp32)
// piece products per product.
//
// Measured, train steps on a GB300, one batched contraction per launch (33 launches
// per slice, every intermediate through memory) against these kernels: [4,12,8192]
// fp32 relu, d = 64, M = 128, C = 512 10.17 -> 5.02 ms; non-causal [8,8,4096] bf16, d = 64,
// M = 256 5.97 -> 2.28 ms; [1,4,65536] bf16, d = 128, M = 256, C = 16 30.05 -> 9.18 ms;
// [1,1,256] fp32, d = 16, M = 32 843 -> 50 us.
#pragma once
#include "simt_tiles.h"
#include "tile_math.cuh"

namespace slim {
namespace simt {

constexpr int kChunk = 32;     // features staged at a time by the row kernels

// x . omega as a compensated dot product (FMA TwoProduct and TwoSum, about 48
// bits; Ogita, Rump and Oishi's Dot2): decides ReLU's branch where the
// projection's own error could.
template <typename IO>
__device__ __noinline__ float dot2(const IO* x, const float* om, int d) {
  float sh = 0.f, sl = 0.f;
  for (int j = 0; j < d; ++j) {
    const float xw = Io<IO>::load(x, j), ow = om[j];
    const float p = __fmul_rn(xw, ow), ep = __fmaf_rn(xw, ow, -p);
    float t, e;
    two_sum(sh, p, t, e);
    sh = t;
    sl = __fadd_rn(sl, __fadd_rn(e, ep));
  }
  return __fadd_rn(sh, sl);
}

// g(x)_f from the projection `dot` of row x (global, for ReLU's recheck).  The
// recheck bound covers the accumulation of the 6 (3) piece products over d / 16
// MMA steps, each step's truncation taken as 2^-23 of |omega| |x|, with a
// factor of 2 to spare.
// rowc: row_const of the row.
template <typename IO>
__device__ __forceinline__ float feature_value(const TileArgs& A, float dot, float rowc, int f,
                                               const IO* x, int d) {
  if (A.feature == SLIM_FEAT_EXP) return expf(dot - rowc) * A.inv_sqrt_m;
  if (fabsf(dot) <= A.om_norm[f] * rowc) dot = dot2<IO>(x, A.omega + (size_t)f * d, d);
  return dot > 0.f ? dot * A.inv_sqrt_m : 0.f;
}
// 0.5 |x|^2 for the exponential map; for ReLU the row's factor of the recheck bound
__device__ __forceinline__ float row_const(const TileArgs& A, float half_norm, int d) {
  return A.feature == SLIM_FEAT_RELU ? 4.f * (float)(d + 2) * 5.9604645e-08f * sqrtf(2.f * half_norm)
                                     : half_norm;
}

// A frame is the 64 rows a CTA works on: one tile of 48 or 64 rows, two of 32
// or four of 16 (each padded from its A.pitch rows to A.rows).
struct Frame {
  int c, t0, left;  // chain, first tile, rows of the slice (of the sequence when a frame has
                    // several tiles) from the frame's first on
  size_t row0;      // first row in a caller tensor
};
__device__ __forceinline__ Frame frame_pos(const TileArgs& A, int frame) {
  Frame f;
  f.c = frame / A.nf;
  f.t0 = frame % A.nf * A.per;
  const int sl = f.t0 / A.slice_tiles, w = (f.t0 - sl * A.slice_tiles) * A.pitch, off = sl * A.slice + w;
  f.left = A.b - off;
  if (A.per == 1) f.left = min(f.left, A.slice - w);
  f.row0 = (size_t)f.c * A.L + A.a + off;
  return f;
}
// caller row (from the frame's first) of frame row r, -1 for a padding row
__device__ __forceinline__ int frame_row(const TileArgs& A, const Frame& f, int r) {
  const int i = r >> A.shift, rr = r - (i << A.shift), x = i * A.pitch + rr;
  return rr < A.pitch && x < f.left ? x : -1;
}

// The frame's rows of one caller tensor (src: its first row; padding rows are
// zero) as pieces [NX][64][D + 8]; row_c (when given): row_const per row.
// D / 8 neighbouring lanes share a row.
template <typename IO, int D>
__device__ __forceinline__ void load_rows(const TileArgs& A, const Frame& f, const IO* src, bf16* dst,
                                          float* row_c) {
  constexpr int NX = Pieces<IO>::NX, PD = D + 8, G = D / 8;
  for (int e = threadIdx.x; e < kTile * G; e += kThreads) {
    const int r = e / G, c8 = (e % G) * 8, x = frame_row(A, f, r);
    float v[8] = {};
    if (x >= 0) load8(src + (size_t)x * D + c8, v);
    store_pieces8<NX>(dst + r * PD + c8, kTile * PD, v);
    if (row_c) {
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) s = fmaf(v[i], v[i], s);
#pragma unroll
      for (int o = 1; o < G; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (c8 == 0) row_c[r] = row_const(A, 0.5f * s, D);
    }
  }
}

// ------------------------------------------------------------------ FMA projections
// The forward's features (and the backward's of fp32 problems with d <= 32) come
// from fp32 FMAs, one per term in j order: an MMA's truncating sum of 16 products
// is a few times less exact, which the exponential passes on whole.  A CTA
// projects 64 rows onto W = 64 or 32 features at a time; a thread has rows rt,
// rt + 16, rt + 32, rt + 48 and W / 16 neighbouring features, 16 FMAs per
// feature for every 4 + W / 16 16-byte (8-byte) shared-memory reads, which is
// bound by the FMA issue rate for W = 64.
template <int D>
constexpr int fp_pitch() { return D + 4; }  // floats: 4 neighbouring rows fall into 4 bank groups

// fp32 rows of a frame and their |x|^2 (summed as one warp's lanes do: strided
// terms, then a butterfly); needs a __syncthreads before the rows are read.
template <typename IO, int D>
__device__ __forceinline__ void load_rows_fp(const TileArgs& A, const Frame& f, const IO* src, float* xs) {
  constexpr int G = D / 8, XP = fp_pitch<D>();
  for (int e = threadIdx.x; e < kTile * G; e += kThreads) {
    const int r = e / G, c8 = (e % G) * 8, x = frame_row(A, f, r);
    float v[8] = {};
    if (x >= 0) load8(src + (size_t)x * D + c8, v);
    float4* d = reinterpret_cast<float4*>(xs + r * XP + c8);
    d[0] = make_float4(v[0], v[1], v[2], v[3]);
    d[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
}
template <int D>
__device__ __forceinline__ void row_norms(const float* xs, float* norm2) {
  for (int r = threadIdx.x / 32; r < kTile; r += kThreads / 32) {
    const float s = warp_norm2<D>(xs + r * fp_pitch<D>());
    if (threadIdx.x % 32 == 0) norm2[r] = s;
  }
}
// W features of Omega, columns c0.. of its [M / 64][D][64] layout, to [D][W]
template <int D, int W>
__device__ __forceinline__ void stage_omega(float* dst, const float* om_t, int c0) {
  const float* src = om_t + (size_t)(c0 / 64) * D * 64 + c0 % 64;
  for (int e = threadIdx.x; e < D * W / 4; e += kThreads) {
    const int j = e / (W / 4), q = (e % (W / 4)) * 4;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + j * W + q)),
                 "l"(src + (size_t)j * 64 + q)
                 : "memory");
  }
}
// g of the frame's 64 rows at features c0 .. c0 + W - 1 (0 in padding rows and
// past M); put(row, feature offset, W / 16 values) stores them.
// NI: the row groups (16 rows) to compute; the rest of the frame gets 0.
template <int D, int W, int NI, typename Put>
__device__ __forceinline__ void features_rows(const TileArgs& A, const Frame& f, const float* xs,
                                            const float* norm2, const float* om, int c0, Put put) {
  constexpr int XP = fp_pitch<D>(), NF = W / 16;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int fq = ((warp & 1) * 8 + lane % 8) * NF, rt = (warp >> 1) * 4 + lane / 8;
  float acc[NI][NF] = {};
  if (A.feature == SLIM_FEAT_SQUARE) {
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int n = 0; n < NF; ++n)
        if (c0 + fq + n < D) {
          const float x = xs[(rt + 16 * i) * XP + c0 + fq + n];
          acc[i][n] = x * x;
        }
  } else {
#pragma unroll 4
    for (int j = 0; j < D; j += 4) {
      float x[NI][4], o[4][NF];
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(xs + (rt + 16 * i) * XP + j);
        x[i][0] = v.x; x[i][1] = v.y; x[i][2] = v.z; x[i][3] = v.w;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (NF == 4) {
          const float4 v = *reinterpret_cast<const float4*>(om + (j + k) * W + fq);
          o[k][0] = v.x; o[k][1] = v.y; o[k][NF - 2] = v.z; o[k][NF - 1] = v.w;
        } else {
          const float2 v = *reinterpret_cast<const float2*>(om + (j + k) * W + fq);
          o[k][0] = v.x; o[k][1] = v.y;
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
          for (int n = 0; n < NF; ++n) acc[i][n] = fmaf(x[i][k], o[k][n], acc[i][n]);
    }
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int r = rt + 16 * i;
      const bool ok = frame_row(A, f, r) >= 0;
      const float n2 = norm2[r];
#pragma unroll
      for (int n = 0; n < NF; ++n) {
        const int m = c0 + fq + n;
        acc[i][n] = ok && m < A.M
                        ? feature_fp<D>(A.feature, acc[i][n], n2, A.feature == SLIM_FEAT_RELU ? A.om_norm[m] : 0.f,
                                        A.inv_sqrt_m, xs + r * XP, om + fq + n, W)
                        : 0.f;
      }
    }
  }
#pragma unroll
  for (int i = 0; i < NI; ++i) put(rt + 16 * i, fq, acc[i]);
  const float zero[NF] = {};
#pragma unroll
  for (int i = NI; i < 4; ++i) put(rt + 16 * i, fq, zero);
}
// A frame whose rows all lie in its first 16 (a few new rows on a running state)
// projects those alone; HALF: so does one whose rows lie in its first 32 (k_out_short on
// one slice of 17 to 32 rows, d = 128, M = 256: 61 -> 47 us with its second tile left out
// too; in every kernel that variant cost 1 % of the C = 16 and quadratic steps).
template <int D, int W, bool HALF = false, typename Put>
__device__ __forceinline__ void features_fp(const TileArgs& A, const Frame& f, const float* xs,
                                            const float* norm2, const float* om, int c0, Put put) {
  if (f.left <= (A.pitch < 16 ? A.pitch : 16))
    features_rows<D, W, 1>(A, f, xs, norm2, om, c0, put);
  else if (HALF && f.left <= (A.pitch < 32 ? A.pitch : 32))
    features_rows<D, W, 2>(A, f, xs, norm2, om, c0, put);
  else
    features_rows<D, W, 4>(A, f, xs, norm2, om, c0, put);
}

constexpr int kPF = 64 + 8;  // row pitch of the forward's 64 x 64 chunk tiles

// features_fp into pieces [NS][64][kPF]
template <int D, int NS, bool HALF = false>
__device__ __forceinline__ void features_to_pieces(const TileArgs& A, const Frame& f, const float* xs,
                                                   const float* norm2, const float* om, int c0,
                                                   bf16* dst) {
  features_fp<D, 64, HALF>(A, f, xs, norm2, om, c0, [&](int r, int fo, const float(&v)[4]) {
    uint32_t a[NS], b[NS];
    split_pair<NS>(v[0], v[1], a);
    split_pair<NS>(v[2], v[3], b);
#pragma unroll
    for (int p = 0; p < NS; ++p)
      *reinterpret_cast<uint2*>(dst + (p * 64 + r) * kPF + fo) = make_uint2(a[p], b[p]);
  });
}

// ------------------------------------------------------------------ Delta_t
// One CTA per frame (several where frames are few, see run_delta): g(K) and, tile by tile,
// Delta_t = g(K)^T [V | 1].  Features
// are taken 64 at a time: project (FMA pipe), split into pieces in shared memory,
// then the tile products from there.  g(K)'s pieces are kept for the kernels that
// read the frame's keys.  The z column (sum of g(K) over the tile's rows) is a
// running fp32 sum in row order for d >= 64 and a column of ones in the MMAs
// otherwise.  The tiles of a frame of short ones are added up here, in order, as a
// value/error pair: a state is 132 KB for d = 128, M = 256, and one per 16 rows through
// global memory (written, scanned, read back) was most of the C = 16 step.  k_out_short
// forms the states inside the frame again.
// Forward and backward call this kernel on the same tiles, so the backward's
// rollback subtracts exactly what the forward added.
// Bound by issue (44 %) and the projection's shared-memory reads (0.5 floats per FMA;
// l1tex 54 %): 768 frames of d = 64, M = 128 in fp32 take 76 us.
template <typename IO, int D>
struct DeltaSmem {
  static constexpr int NX = Pieces<IO>::NX, NS = Pieces<IO>::NS, PD = D + 8;
  static constexpr int xs = kTile * fp_pitch<D>() * 4, om = D * 64 * 4, v = NX * kTile * PD * 2,
                       ph = NS * 64 * kPF * 2;
  static constexpr int bytes = xs + om + v + ph + kTile * 4 + 4 * 64 * 4;
  // three CTAs on an SM for bf16 where their shared memory fits (228 KB, 1 KB of it per
  // CTA): 482 -> 465 us of the non-causal step; fp32 spills (ragged step 378 -> 388 us)
  static constexpr int ctas = NX == 1 && 3 * (bytes + 1024) <= 233472 ? 3 : 2;
  static_assert(bytes <= kSmemMax, "shared memory");
};

template <typename IO, int D>
__global__ void __launch_bounds__(kThreads, (DeltaSmem<IO, D>::ctas)) k_delta(const __grid_constant__ TileArgs A) {
  using S = DeltaSmem<IO, D>;
  constexpr int NX = S::NX, NS = S::NS, PD = S::PD;
  constexpr int CW = D >= 32 ? D / 2 : 16, NB = CW / 8;  // columns of a warp
  extern __shared__ uint4 smem_raw[];
  float* xs = reinterpret_cast<float*>(smem_raw);
  float* om = xs + S::xs / 4;
  bf16* Vs = reinterpret_cast<bf16*>(om + S::om / 4);
  bf16* Ph = Vs + S::v / 2;
  float* norm2 = reinterpret_cast<float*>(Ph + S::ph / 2);
  float* zt = norm2 + kTile;  // [tile][64]
  const int frame = blockIdx.x;
  const Frame f = frame_pos(A, frame);
  const bool square = A.feature == SLIM_FEAT_SQUARE;
  // the caller's rows before the kernel ahead is waited for (see launch_pdl)
  load_rows_fp<IO, D>(A, f, static_cast<const IO*>(A.k) + f.row0 * D, xs);
  load_rows<IO, D>(A, f, static_cast<const IO*>(A.v) + f.row0 * D, Vs, nullptr);
  __syncthreads();
  row_norms<D>(xs, norm2);
  pdl_wait();
  pdl_launch();
  const int cstep = 64 * gridDim.y;  // a frame's chunks may be dealt to several CTAs
  if (!square) {
    stage_omega<D, 64>(om, A.om_t, 64 * blockIdx.y);
    cp_commit();
  }

  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, g = lane >> 2, t = lane & 3;
  const int fb = warp & 3, h = warp >> 2;  // 16 features of the chunk, half of the columns
  const int ksteps = A.rows / 16;          // k16 steps per tile
  // two reduction groups (even and odd steps) for few features
  const bool two = A.rows == 64 && (A.M == 32 || (A.M == 16 && NS == 3));
  // a tile's total, or (several tiles) the frame's pair: values, then errors
  float* dl = A.delta + (A.per == 1 ? (size_t)frame : 2 * (size_t)frame) * A.E;
  float* zd = A.per == 1 ? dl + A.M * D : A.zdelta + ((size_t)f.c * A.nt + f.t0) * A.M;
  bf16* pk = A.phi_k ? A.phi_k + (size_t)frame * NS * 64 * A.M : nullptr;
  const int ntl = min(A.per, A.nt - f.t0);  // tiles of this frame
  for (int c0 = 64 * blockIdx.y; c0 < A.M; c0 += cstep) {
    cp_wait<0>();
    __syncthreads();
    features_to_pieces<D, NS>(A, f, xs, norm2, om, c0, Ph);
    __syncthreads();
    if (!square && c0 + cstep < A.M) {
      stage_omega<D, 64>(om, A.om_t, c0 + cstep);
      cp_commit();
    }
    const int nf = min(64, A.M - c0);
    if (pk)
      for (int e = tid; e < 64 * (nf / 8); e += kThreads) {
        const int r = e / (nf / 8), c8 = (e % (nf / 8)) * 8;
#pragma unroll
        for (int p = 0; p < NS; ++p)
          *reinterpret_cast<uint4*>(pk + ((size_t)p * 64 + r) * A.M + c0 + c8) =
              *reinterpret_cast<const uint4*>(Ph + (p * 64 + r) * kPF + c8);
      }
    if (16 * fb < nf) {
      const int f0 = c0 + 16 * fb + g;
      float a0[NB][4] = {}, a1[NB][4] = {}, lo[NB][4] = {}, z0[4] = {}, z1[4] = {}, zlo[4] = {};
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        const int i = 16 * ks >> A.shift, last = ks == ksteps * (i + 1) - 1;
        if (ks >= ksteps * ntl) break;
        uint32_t a[NS][4];
        ld_at<NS>(a, Ph, 64 * kPF, kPF, 16 * fb, 16 * ks);
        const bool g1 = two && (ks & 1);
        if (D >= 32 || h == 0) {
#pragma unroll
          for (int nb = 0; nb < NB / 2; ++nb) {
            uint32_t b[NX][4];
            ld_bt<NX>(b, Vs, kTile * PD, PD, (D >= 32 ? CW * h : 0) + 16 * nb, 16 * ks);
            if (g1)
              mma_pieces<NS, NX>(a1[2 * nb], a1[2 * nb + 1], a, b);
            else
              mma_pieces<NS, NX>(a0[2 * nb], a0[2 * nb + 1], a, b);
          }
        }
        if (D < 64 && h == 1) {
          const uint32_t one = g == 0 ? kOnes : 0u;
          if (g1)
            mma_n8<NS>(z1, a, one, one);
          else
            mma_n8<NS>(z0, a, one, one);
        }
        if (last) {
          if (D >= 32 || h == 0) {
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) {
              float* dst = dl + (size_t)f0 * D + (D >= 32 ? CW * h : 0) + 8 * nb + 2 * t;
              if (A.per > 1) {  // a1: the pair's value, lo its error
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  pair_add(a1[nb][c], lo[nb][c], a0[nb][c]);
                  a0[nb][c] = 0.f;
                }
                if (i + 1 < ntl) continue;
                *reinterpret_cast<float2*>(dst) = make_float2(a1[nb][0], a1[nb][1]);
                *reinterpret_cast<float2*>(dst + 8 * D) = make_float2(a1[nb][2], a1[nb][3]);
                *reinterpret_cast<float2*>(dst + A.E) = make_float2(lo[nb][0], lo[nb][1]);
                *reinterpret_cast<float2*>(dst + A.E + 8 * D) = make_float2(lo[nb][2], lo[nb][3]);
              } else {
                if (two)
#pragma unroll
                  for (int c = 0; c < 4; ++c) a0[nb][c] += a1[nb][c];
                *reinterpret_cast<float2*>(dst) = make_float2(a0[nb][0], a0[nb][1]);
                *reinterpret_cast<float2*>(dst + 8 * D) = make_float2(a0[nb][2], a0[nb][3]);
              }
            }
          }
          if (D < 64 && h == 1) {
            if (two)
#pragma unroll
              for (int c = 0; c < 4; ++c) z0[c] += z1[c];
            if (t == 0) {
              zd[(size_t)i * A.M + f0] = z0[0];
              zd[(size_t)i * A.M + f0 + 8] = z0[2];
            }
            if (A.per > 1) {
#pragma unroll
              for (int c = 0; c < 4; c += 2) pair_add(z1[c], zlo[c], z0[c]);
              if (i + 1 == ntl && t == 0) {
                float* dz = dl + A.M * D + f0;
                dz[0] = z1[0];
                dz[8] = z1[2];
                dz[A.E] = zlo[0];
                dz[A.E + 8] = zlo[2];
              }
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) z0[c] = 0.f;
          }
        }
      }
    }
    if (D >= 64) {  // z: a lane sums two neighbouring features over one tile's rows
      const int i = (warp - (c0 / 64) * A.per) & 7;  // the duty moves from warp to warp
      if (i < ntl && 2 * lane < nf) {
        const bf16* p = Ph + (size_t)i * A.rows * kPF + 2 * lane;
        float s[2][2] = {};
        for (int k0 = 0; k0 < A.rows; k0 += 16) {
          const bool g1 = two && (k0 & 16);
          float x = g1 ? s[1][0] : s[0][0], y = g1 ? s[1][1] : s[0][1];
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            float2 v = make_float2(0.f, 0.f);
#pragma unroll
            for (int q = NS - 1; q >= 0; --q) {
              const float2 w = unpack2(*reinterpret_cast<const uint32_t*>(p + (q * 64 + k0 + k) * kPF));
              v.x += w.x;
              v.y += w.y;
            }
            x += v.x;
            y += v.y;
          }
          if (g1) {
            s[1][0] = x;
            s[1][1] = y;
          } else {
            s[0][0] = x;
            s[0][1] = y;
          }
        }
        if (two) {
          s[0][0] += s[1][0];
          s[0][1] += s[1][1];
        }
        *reinterpret_cast<float2*>(zd + (size_t)i * A.M + c0 + 2 * lane) = make_float2(s[0][0], s[0][1]);
        if (A.per > 1) *reinterpret_cast<float2*>(zt + i * 64 + 2 * lane) = make_float2(s[0][0], s[0][1]);
      }
      if (A.per > 1) {  // the frame's pair
        __syncthreads();
        if (tid < nf) {
          float zh = 0.f, zl = 0.f;
          for (int i = 0; i < ntl; ++i) pair_add(zh, zl, zt[i * 64 + tid]);
          dl[A.M * D + c0 + tid] = zh;
          dl[A.E + A.M * D + c0 + tid] = zl;
        }
      }
    }
  }
}

// A chunk (up to R rows) of a state's S (fp32 rows of D) on its way to shared
// memory as pieces: held in registers between load and store, so that the loads
// overlap a chunk's products.
template <int D, int R>
struct StateChunk {
  static constexpr int N = (R * D / 8 + kThreads - 1) / kThreads;
  float v[N][8];
  __device__ __forceinline__ void load(const float* S, int rows) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int e = threadIdx.x + i * kThreads;
      if (e < rows * (D / 8)) load8(S + (size_t)e * 8, v[i]);
    }
  }
  // SWZ: rows of D elements without padding, their 16-byte chunks swizzled by the row
  template <int NP, bool SWZ = false>
  __device__ __forceinline__ void store(bf16* dst, int rows) const {
    constexpr int P = SWZ ? D : D + 8;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int e = threadIdx.x + i * kThreads, r = e / (D / 8), c = e % (D / 8);
      if (e < rows * (D / 8)) store_pieces8<NP>(dst + r * P + (SWZ ? c ^ (r & 7) : c) * 8, R * P, v[i]);
    }
  }
};
// ld_bt of 64 rows that StateChunk stored
template <int NP, int D, bool SWZ>
__device__ __forceinline__ void ld_state(uint32_t (&b)[NP][4], const bf16* p, int n0, int k0) {
  if (!SWZ) {
    ld_bt<NP>(b, p, 64 * (D + 8), D + 8, n0, k0);
    return;
  }
  const int l = threadIdx.x & 31, r = k0 + (l & 15), c = n0 / 8 + (l >> 4);
  p += r * D + (c ^ (r & 7)) * 8;
#pragma unroll
  for (int i = 0; i < NP; ++i) ldsm4t(b[i], p + i * 64 * D);
}

// `rows` rows of W bf16 (W % 8 == 0) in NP pieces, global row pitch gp and piece
// stride gs, to shared memory (pitch sp, piece stride ss), asynchronously.
template <int NP>
__device__ __forceinline__ void stage_rows(bf16* dst, int ss, int sp, const bf16* src, size_t gs,
                                           int gp, int rows, int W) {
  const int u = W / 8, n = rows * u;
  for (int e = threadIdx.x; e < n; e += kThreads) {
    const int r = e / u, c8 = (e % u) * 8;
#pragma unroll
    for (int p = 0; p < NP; ++p) cp16(dst + p * ss + r * sp + c8, src + p * gs + (size_t)r * gp + c8);
  }
}

// ------------------------------------------------------------------ readout
// One CTA per frame: g(Q), A = tril(g(Q) g(K)^T) inside each tile, out = (g(Q) S +
// A V) / (g(Q) z + A 1).  k_out: one tile of 48 or 64 rows.  Warp (r, h) has rows 16 r ..
// 16 r + 15 and the h-th half of every product's columns.  The next chunk's Omega and
// state travel while this one's products run, its g(K) while it is projected; FMA and
// tensor pipe overlap across the two CTAs of an SM.  Bound by issue and the latency of a
// chunk's phases (44 % issue, 19 % tensor pipe at d = 64 in fp32); 768 frames of d = 64,
// M = 128 in fp32 take 96 us, 142 us with one CTA on an SM (the state chunk padded).
template <typename IO, int D>
struct OutSmem {
  static constexpr int NX = Pieces<IO>::NX, NS = Pieces<IO>::NS, PD = D + 8;
  // d = 64 in fp32: a padded state chunk would leave room for one CTA on an SM
  static constexpr bool SWZ = D == 64 && NX == 3;
  static constexpr int xs = kTile * fp_pitch<D>() * 4, om = D * 64 * 4, ph = NS * 64 * kPF * 2,
                       ps = NS * 64 * (SWZ ? D : PD) * 2, zs = 64 * 4;
  static constexpr int bytes = xs + om + 2 * ph + ps + zs + 2 * kTile * 4;
  static_assert(D > 64 || 2 * (bytes + 1024) <= 233472, "two CTAs on an SM");
  static_assert(NX * kTile * PD * 2 <= xs + om, "V in the projections' buffers");
  static_assert(bytes <= kSmemMax, "shared memory");
};

template <typename IO, int D>
__global__ void __launch_bounds__(kThreads, D <= 64 ? 2 : 1)
    k_out(const __grid_constant__ TileArgs A) {
  using S = OutSmem<IO, D>;
  constexpr int NX = S::NX, NS = S::NS, PD = S::PD;
  constexpr int CW = D >= 32 ? D / 2 : 16, NB = CW / 8;       // columns of a warp
  constexpr bool ZM = D < 64;                                 // den as an MMA column
  extern __shared__ uint4 smem_raw[];
  float* xs = reinterpret_cast<float*>(smem_raw);
  float* om = xs + S::xs / 4;
  bf16* Ph = reinterpret_cast<bf16*>(om + S::om / 4);
  bf16* Kp = Ph + S::ph / 2;
  bf16* Ps = Kp + S::ph / 2;
  float* zs = reinterpret_cast<float*>(Ps + S::ps / 2);  // z rounded to the pieces
  float* norm2 = zs + 64;
  float* den_s = norm2 + kTile;
  bf16* Vs = reinterpret_cast<bf16*>(xs);
  const int frame = blockIdx.x;
  const Frame f = frame_pos(A, frame);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, g = lane >> 2, t = lane & 3;
  const int h = warp >> 2, r = warp & 3, r0 = 16 * r;
  const size_t MD = (size_t)A.M * D;
  const float* Pt = A.P + f.c * A.p_chain + f.t0 * A.p_frame;
  const bf16* pk = A.phi_k + (size_t)frame * NS * 64 * A.M;
  const bool square = A.feature == SLIM_FEAT_SQUARE;
  const int cb = D >= 32 ? CW * h : 0;                    // first column
  const bool cols = D >= 32 || h == 0;
  const int k0 = 32 * h;                                  // first key of this warp's scores

  StateChunk<D, 64> pc;
  auto stage_keys = [&](int c0) {
    if (A.causal)
      stage_rows<NS>(Kp, 64 * kPF, kPF, pk + c0, (size_t)64 * A.M, A.M, 64, min(64, A.M - c0));
    cp_commit();
  };
  auto stage_om = [&](int c0) {
    if (!square) stage_omega<D, 64>(om, A.om_t, c0);
    cp_commit();
  };
  // all but the state comes from the caller or from kernels before the one ahead
  stage_om(0);
  stage_keys(0);
  load_rows_fp<IO, D>(A, f, static_cast<const IO*>(A.q) + f.row0 * D, xs);
  __syncthreads();
  row_norms<D>(xs, norm2);
  pdl_wait();
  pdl_launch();
  pc.load(Pt, min(64, A.M));
  pc.template store<NS, S::SWZ>(Ps, min(64, A.M));

  float num[NB][4] = {}, sc[4][4] = {}, dz[4] = {}, de = 0.f;
  // the warps with the fewest scores sum den for d >= 64, a row per lane
  const int dr = warp == 4 ? lane : warp == 5 ? 32 + lane : -1;
  for (int c0 = 0; c0 < A.M; c0 += 64) {
    const int nf = min(64, A.M - c0);
    cp_wait<1>();
    __syncthreads();
    features_to_pieces<D, NS>(A, f, xs, norm2, om, c0, Ph);
    if (!ZM && tid < nf) zs[tid] = round_pieces<NS>(Pt[MD + c0 + tid]);
    cp_wait<0>();
    __syncthreads();
    const bool more = c0 + 64 < A.M;
    if (more) stage_om(c0 + 64);
    if (more) pc.load(Pt + (size_t)(c0 + 64) * D, min(64, A.M - c0 - 64));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (16 * i >= nf) break;
      uint32_t a[NS][4];
      ld_a<NS>(a, Ph, 64 * kPF, kPF, r0, 16 * i);
      if (cols) {
#pragma unroll
        for (int nb = 0; nb < NB / 2; ++nb) {
          uint32_t b[NS][4];
          ld_state<NS, D, S::SWZ>(b, Ps, cb + 16 * nb, 16 * i);
          mma_pieces<NS, NS>(num[2 * nb], num[2 * nb + 1], a, b);
        }
      }
      if (ZM && h == 1) {  // the z column
        uint32_t w0[NS] = {}, w1[NS] = {};
        if (g == 0) {
          const float* z = Pt + MD + c0 + 16 * i + 2 * t;
          split_pair<NS>(z[0], z[1], w0);
          split_pair<NS>(z[8], z[9], w1);
        }
#pragma unroll
        for (int o = NS - 1; o >= 0; --o)
#pragma unroll
          for (int x = 0; x <= o; ++x) mma16816(dz, a[x], w0[o - x], w1[o - x]);
      }
      if (A.causal) {
#pragma unroll
        for (int kb = 0; kb < 2; ++kb)
          if (k0 + 16 * kb <= r0) {  // later keys are masked
            uint32_t b[NS][4];
            ld_b<NS>(b, Kp, 64 * kPF, kPF, k0 + 16 * kb, 16 * i);
            mma_pieces<NS, NS>(sc[2 * kb], sc[2 * kb + 1], a, b);
          }
      }
      if (!ZM && dr >= 0) {  // den += g(q) z, feature after feature
#pragma unroll
        for (int k = 0; k < 16; k += 8) {
          float x[8];
          add_pieces8<NS>(Ph + dr * kPF + 16 * i + k, 64 * kPF, x);
#pragma unroll
          for (int u = 0; u < 8; ++u) de = fmaf(x[u], zs[16 * i + k + u], de);
        }
      }
    }
    __syncthreads();
    if (more) {
      stage_keys(c0 + 64);
      pc.template store<NS, S::SWZ>(Ps, min(64, A.M - c0 - 64));
    }
  }
  if (A.causal) {
    // masked scores as pieces (in g(Q)'s place), then A [V | 1]
#pragma unroll
    for (int kb = 0; kb < 4; ++kb)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int row = r0 + g + 8 * hf, key = k0 + 8 * kb + 2 * t;
        uint32_t w[NS];
        split_pair<NS>(key <= row ? sc[kb][2 * hf] : 0.f, key + 1 <= row ? sc[kb][2 * hf + 1] : 0.f, w);
#pragma unroll
        for (int p = 0; p < NS; ++p)
          *reinterpret_cast<uint32_t*>(Ph + (p * 64 + row) * kPF + key) = w[p];
      }
    load_rows<IO, D>(A, f, static_cast<const IO*>(A.v) + f.row0 * D, Vs, nullptr);
    __syncthreads();
    float av[NB][4] = {}, az[4] = {};
#pragma unroll
    for (int kb = 0; kb < 4; ++kb)
      if (kb <= r) {
        uint32_t a[NS][4];
        ld_a<NS>(a, Ph, 64 * kPF, kPF, r0, 16 * kb);
        if (cols) {
#pragma unroll
          for (int nb = 0; nb < NB / 2; ++nb) {
            uint32_t b[NX][4];
            ld_bt<NX>(b, Vs, kTile * PD, PD, cb + 16 * nb, 16 * kb);
            mma_pieces<NS, NX>(av[2 * nb], av[2 * nb + 1], a, b);
          }
        }
        if (ZM && h == 1) {
          const uint32_t one = g == 0 ? kOnes : 0u;
          mma_n8<NS>(az, a, one, one);
        }
      }
#pragma unroll
    for (int nb = 0; nb < NB; ++nb)
#pragma unroll
      for (int c = 0; c < 4; ++c) num[nb][c] = av[nb][c] + num[nb][c];
#pragma unroll
    for (int c = 0; c < 4; ++c) dz[c] = az[c] + dz[c];
    if (!ZM && dr >= 0) {
      float e = 0.f;
      for (int k = 0; k <= dr; k += 8) {
        float x[8];
        add_pieces8<NS>(Ph + dr * kPF + k, 64 * kPF, x);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (k + u <= dr) e += x[u];
      }
      de = e + de;
    }
  }
  if (ZM) {
    if (h == 1 && t == 0) {
      den_s[r0 + g] = dz[0];
      den_s[r0 + g + 8] = dz[2];
    }
  } else if (dr >= 0) {
    den_s[dr] = de;
  }
  __syncthreads();
  if (!cols) return;
  IO* og = static_cast<IO*>(A.o) + f.row0 * D;
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    const int row = r0 + g + 8 * hf, x = frame_row(A, f, row);
    const float den = den_s[row];
    if (x >= 0) {
#pragma unroll
      for (int nb = 0; nb < NB; ++nb)
        store2(og + (size_t)x * D + cb + 8 * nb + 2 * t, den != 0.f ? num[nb][2 * hf] / den : 0.f,
               den != 0.f ? num[nb][2 * hf + 1] / den : 0.f);
    }
  }
}

// k_out for frames of several short tiles (two of 32 rows, four of 16).  The state
// moves on from tile to tile inside the frame: a warp owns 16 columns of a chunk's
// state, as a value/error pair in registers from the chunk's start (k_carry's
// pair), and after each tile's readout adds the tile's Delta^T = V^T g(K) from an MMA, in
// the layout of the readout's B fragments.  Products over the features sum their k16
// steps in A.ks_n (readout) and A.ks_a (scores) interleaved groups, added in order
// at the end.  Where the columns leave half of the warps free (d = 64 and less) two
// warps share a column block, each with every other k16 step.  Scores, den and masks as
// in k_out, warp (r, h) with rows 16 r .. 16 r + 15 and half of the tile's keys.
// CAUSAL false: the non-causal readout, all tiles from one state, absent tiles left out; two
// CTAs on an SM where they fit (600 chains of 9 rows, d = 64, M = 128, bf16: 139 -> 106 us for the
// whole forward; as an argument of the causal kernel the same cost its C = 16 step 0.4 %).
template <typename IO, int D, bool CAUSAL>
struct ShortSmemOut {
  static constexpr int NX = Pieces<IO>::NX, NS = Pieces<IO>::NS, PD = D + 8;
  static constexpr int xs = kTile * fp_pitch<D>() * 4, om = D * 64 * 4, ph = NS * 64 * kPF * 2,
                       kp = CAUSAL ? ph : 0, v = CAUSAL ? NX * kTile * PD * 2 : 0, zs = 4 * 64 * 4;
  static constexpr int bytes = xs + om + ph + kp + v + zs + 2 * kTile * 4;
  static constexpr int NCB = D / 16, NH = D == 128 ? 1 : 2;
  static_assert(NH == 1 || NCB * 32 * 64 * 4 <= xs + om, "the second halves' sums");
  static_assert(bytes <= kSmemMax, "shared memory");
  // without scores and state products two CTAs fit an SM; for d < 64, and for bf16 at
  // d = 128, they would spill (17 chains of 216 rows, C = 7, d = 128: 130 us against 114)
  static constexpr int ctas = !CAUSAL && (D == 64 || (D == 128 && NX == 3)) ? 2 : 1;
  static_assert(ctas == 1 || 2 * (bytes + 1024) <= 233472, "two CTAs on an SM");
};

template <typename IO, int D, int MODE, bool CAUSAL>
__global__ void __launch_bounds__(kThreads, (ShortSmemOut<IO, D, CAUSAL>::ctas)) k_out_short(const __grid_constant__ TileArgs A) {
  using S = ShortSmemOut<IO, D, CAUSAL>;
  constexpr int NX = S::NX, NS = S::NS, PD = S::PD, NCB = S::NCB, NH = S::NH;
  constexpr int GN = NH == 1 && MODE == 2 && NS == 2 ? 4 : 2;          // readout groups of a warp, at most
  constexpr int GA = MODE == 1 ? 2 : NS == 2 ? 8 : 4;                  // score groups, at most
  constexpr int KB = MODE == 1 ? 2 : 1;                                // n8 blocks of a warp's scores
  constexpr int NTI = MODE == 1 ? 2 : 4, RB = 4 / NTI;                 // tiles, 16-row groups of a tile
  constexpr bool ZM = D < 64;                                          // den as an MMA column
  extern __shared__ uint4 smem_raw[];
  float* xs = reinterpret_cast<float*>(smem_raw);
  float* om = xs + S::xs / 4;
  bf16* Ph = reinterpret_cast<bf16*>(om + S::om / 4);
  bf16* Kp = Ph + S::ph / 2;
  bf16* Vs = Kp + S::kp / 2;
  float* zs = reinterpret_cast<float*>(Vs + S::v / 2);  // [tile][64]: z (d >= 64: rounded to the pieces)
  float* norm2 = zs + 4 * 64;
  float* den_s = norm2 + kTile;
  const int frame = blockIdx.x;
  const Frame f = frame_pos(A, frame);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, g = lane >> 2, t = lane & 3;
  const int h = warp >> 2, r = warp & 3, r0 = 16 * r;
  const int ti = r / RB;                                  // this warp's tile in the scores
  const int cb = 16 * (warp % NCB), hh = warp / NCB;      // its columns and half in the readout
  const bool halves = NH == 2 && A.ks_n > 1;
  const int ntl = min(A.per, A.nt - f.t0);
  const size_t MD = (size_t)A.M * D;
  const float* Pt = A.P + f.c * A.p_chain + f.t0 / A.per * A.p_frame;
  const long long plo = A.p_lo;                           // from the pair's values to its errors
  const float* zd = A.zdelta + ((size_t)f.c * A.nt + f.t0) * A.M;
  const bf16* pk = A.phi_k + (size_t)frame * NS * 64 * A.M;
  const bool causal = CAUSAL && A.causal;
  const bool square = A.feature == SLIM_FEAT_SQUARE;
  const int k0 = MODE == 1 ? 32 * ti + 16 * h : r0;       // first key of this warp's scores

  auto stage_keys = [&](int c0) {
    if (causal)
      stage_rows<NS>(Kp, 64 * kPF, kPF, pk + c0, (size_t)64 * A.M, A.M, 64, min(64, A.M - c0));
    cp_commit();
  };
  auto stage_om = [&](int c0) {
    if (!square) stage_omega<D, 64>(om, A.om_t, c0);
    cp_commit();
  };
  stage_om(0);
  stage_keys(0);
  load_rows_fp<IO, D>(A, f, static_cast<const IO*>(A.q) + f.row0 * D, xs);
  if (CAUSAL) load_rows<IO, D>(A, f, static_cast<const IO*>(A.v) + f.row0 * D, Vs, nullptr);
  __syncthreads();
  row_norms<D>(xs, norm2);
  pdl_wait();  // the state; the rest is older
  pdl_launch();

  float num[GN][4][2][4] = {}, sc[GA][KB][4] = {}, dz[4][4] = {}, de[4] = {};
  const int dr = warp == 4 ? lane : warp == 5 ? 32 + lane : -1;  // den's rows (d >= 64)
  const float* zrow = zs + (dr < 0 ? 0 : dr / (16 * RB) * 64);
  auto own = [&](int i) { return halves ? hh < 2 && (i & 1) == hh : hh == 0; };
  for (int c0 = 0; c0 < A.M; c0 += 64) {
    const int nf = min(64, A.M - c0);
    // the chunk's state at the frame's start: element i of step s is column cb + g + 8
    // ((i >> 1) & 1), feature c0 + 16 s + 2 t + (i & 1) + 8 (i >> 2)
    float hi[4][8], lo[4][8];
    auto value = [&](int s, int i) { return S::ctas == 1 ? hi[s][i] + lo[s][i] : hi[s][i]; };
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        hi[s][i] = lo[s][i] = 0.f;
        if (own(s) && 16 * s < nf) {
          const float* p = Pt + (size_t)(c0 + 16 * s + 2 * t + (i & 1) + 8 * (i >> 2)) * D + cb + g + 8 * ((i >> 1) & 1);
          if (S::ctas == 1) {
            hi[s][i] = p[0];
            lo[s][i] = p[plo];
          } else {  // at once: 128 registers
            hi[s][i] = p[0] + p[plo];
          }
        }
      }
    cp_wait<1>();
    __syncthreads();
    features_to_pieces<D, NS, MODE == 1>(A, f, xs, norm2, om, c0, Ph);
    if (tid < nf) {  // z at every tile of the frame
      const float* p = Pt + MD + c0 + tid;
      float zh = p[0], zl = p[plo];
#pragma unroll
      for (int j = 0; j < NTI; ++j)
        if (j < ntl) {
          const float z = zh + zl;
          zs[j * 64 + tid] = ZM ? z : round_pieces<NS>(z);
          if (causal) pair_add(zh, zl, zd[(size_t)j * A.M + c0 + tid]);
        }
    }
    cp_wait<0>();
    __syncthreads();
    const bool more = c0 + 64 < A.M;
    if (more) stage_om(c0 + 64);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (16 * s >= nf) break;
      if (own(s)) {
        const int gn = halves ? (A.ks_n == 4 ? s >> 1 : 0) : s & (A.ks_n - 1);
#pragma unroll
        for (int j = 0; j < NTI; ++j) {
          if ((MODE == 1 || !CAUSAL) && j >= ntl) break;
          uint32_t b[NS][4];
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            uint32_t w0[NS], w1[NS];
            split_pair<NS>(value(s, 2 * q), value(s, 2 * q + 1), w0);
            split_pair<NS>(value(s, 4 + 2 * q), value(s, 5 + 2 * q), w1);
#pragma unroll
            for (int p = 0; p < NS; ++p) {
              b[p][2 * q] = w0[p];
              b[p][2 * q + 1] = w1[p];
            }
          }
          float d[2][4] = {};
#pragma unroll
          for (int y = 0; y < RB; ++y) {
            const int rb = j * RB + y;
            uint32_t a[NS][4];
            ld_a<NS>(a, Ph, 64 * kPF, kPF, 16 * rb, 16 * s);
#pragma unroll
            for (int q = 0; q < GN; ++q)
              if (q == gn) mma_pieces<NS, NS>(num[q][rb][0], num[q][rb][1], a, b);
            if (causal && j + 1 < (MODE == 1 ? ntl : NTI)) {  // Delta^T, the pieces' products in Delta's order
              uint32_t v[NX][4], k[NS][4];
              ld_at<NX>(v, Vs, kTile * PD, PD, cb, 16 * rb);
              ld_bt<NS>(k, Kp, 64 * kPF, kPF, 16 * s, 16 * rb);
#pragma unroll
              for (int o = NS - 1; o >= 0; --o)
#pragma unroll
                for (int i = 0; i <= o; ++i)
                  if (o - i < NX) {
                    mma16816(d[0], v[o - i], k[i][0], k[i][1]);
                    mma16816(d[1], v[o - i], k[i][2], k[i][3]);
                  }
            }
          }
          if (causal && j + 1 < (MODE == 1 ? ntl : NTI)) {
#pragma unroll
            for (int i = 0; i < 8; ++i) pair_add(hi[s][i], lo[s][i], d[i >> 2][i & 3]);
          }
        }
      }
      uint32_t a[NS][4];
      ld_a<NS>(a, Ph, 64 * kPF, kPF, r0, 16 * s);
      const int step = c0 / 16 + s, gz = s & (A.ks_n - 1), ga = step & (A.ks_a - 1);
      if (ZM && h == 1) {  // the z column
        uint32_t w0[NS] = {}, w1[NS] = {};
        if (g == 0) {
          const float* z = zs + min(ti, ntl - 1) * 64 + 16 * s + 2 * t;
          split_pair<NS>(z[0], z[1], w0);
          split_pair<NS>(z[8], z[9], w1);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q == gz) {
#pragma unroll
            for (int o = NS - 1; o >= 0; --o)
#pragma unroll
              for (int x = 0; x <= o; ++x) mma16816(dz[q], a[x], w0[o - x], w1[o - x]);
          }
      }
      if (causal) {
        uint32_t b[NS][4];
        if (MODE == 2) {
          ld_b<NS>(b, Kp, 64 * kPF, kPF, r0, 16 * s);
#pragma unroll
          for (int q = 0; q < GA; ++q)
            if (q == ga) {
#pragma unroll
              for (int o = NS - 1; o >= 0; --o)
#pragma unroll
                for (int x = 0; x <= o; ++x)
                  mma16816(sc[q][0], a[x], h ? b[o - x][2] : b[o - x][0], h ? b[o - x][3] : b[o - x][1]);
            }
        } else if (k0 <= r0) {  // later keys are masked
          ld_b<NS>(b, Kp, 64 * kPF, kPF, k0, 16 * s);
#pragma unroll
          for (int q = 0; q < GA; ++q)
            if (q == ga) mma_pieces<NS, NS>(sc[q][0], sc[q][KB - 1], a, b);
        }
      }
      if (!ZM && dr >= 0) {  // den += g(q) z, feature after feature
        float e = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q == gz) e = de[q];
#pragma unroll
        for (int k = 0; k < 16; k += 8) {
          float x[8];
          add_pieces8<NS>(Ph + dr * kPF + 16 * s + k, 64 * kPF, x);
#pragma unroll
          for (int u = 0; u < 8; ++u) e = fmaf(x[u], zrow[16 * s + k + u], e);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q == gz) de[q] = e;
      }
    }
    __syncthreads();
    if (more) stage_keys(c0 + 64);
  }
  // the groups' sums, in order
#pragma unroll
  for (int q = 1; q < 4; ++q)
    if (q < A.ks_n) {
#pragma unroll
      for (int c = 0; c < 4; ++c) dz[0][c] += dz[q][c];
      de[0] += de[q];
    }
  float* red = xs + (warp % NCB) * 32 * 64 + lane;  // [group][32 values] of the second half's warps
  if (halves && hh == 1) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int i = 0; i < 32; ++i) red[(q * 32 + i) * 32] = num[q][i >> 3][(i >> 2) & 1][i & 3];
  }
  if (causal) {
    // masked scores as pieces, in g(Q)'s place
#pragma unroll
    for (int q = 1; q < GA; ++q)
      if (q < A.ks_a) {
#pragma unroll
        for (int kb = 0; kb < KB; ++kb)
#pragma unroll
          for (int c = 0; c < 4; ++c) sc[0][kb][c] += sc[q][kb][c];
      }
#pragma unroll
    for (int kb = 0; kb < KB; ++kb)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int row = r0 + g + 8 * hf, key = k0 + (MODE == 2 ? 8 * h : 8 * kb) + 2 * t;
        uint32_t w[NS];
        split_pair<NS>(key <= row ? sc[0][kb][2 * hf] : 0.f, key + 1 <= row ? sc[0][kb][2 * hf + 1] : 0.f, w);
#pragma unroll
        for (int p = 0; p < NS; ++p)
          *reinterpret_cast<uint32_t*>(Ph + (p * 64 + row) * kPF + key) = w[p];
      }
  }
  __syncthreads();
  if (causal) {
    if (ZM && h == 1) {
      float az[4] = {};
#pragma unroll
      for (int kb = 0; kb < 4; ++kb)
        if (kb <= r && kb / RB == ti) {
          uint32_t a[NS][4];
          ld_a<NS>(a, Ph, 64 * kPF, kPF, r0, 16 * kb);
          const uint32_t one = g == 0 ? kOnes : 0u;
          mma_n8<NS>(az, a, one, one);
        }
#pragma unroll
      for (int c = 0; c < 4; ++c) dz[0][c] = az[c] + dz[0][c];
    }
    if (!ZM && dr >= 0) {
      float e = 0.f;
      for (int k = dr / (16 * RB) * (16 * RB); k <= dr; k += 8) {
        float x[8];
        add_pieces8<NS>(Ph + dr * kPF + k, 64 * kPF, x);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (k + u <= dr) e += x[u];
      }
      de[0] = e + de[0];
    }
  }
  if (ZM) {
    if (h == 1 && t == 0) {
      den_s[r0 + g] = dz[0][0];
      den_s[r0 + g + 8] = dz[0][2];
    }
  } else if (dr >= 0) {
    den_s[dr] = de[0];
  }
  __syncthreads();
  if (hh > 0) return;
  IO* og = static_cast<IO*>(A.o) + f.row0 * D;
#pragma unroll
  for (int rb = 0; rb < 4; ++rb) {
    float av[2][4] = {};
    if (causal) {
#pragma unroll
      for (int kb = 0; kb < 4; ++kb)
        if (kb <= rb && kb / RB == rb / RB) {
          uint32_t a[NS][4], b[NX][4];
          ld_a<NS>(a, Ph, 64 * kPF, kPF, 16 * rb, 16 * kb);
          ld_bt<NX>(b, Vs, kTile * PD, PD, cb, 16 * kb);
          mma_pieces<NS, NX>(av[0], av[1], a, b);
        }
    }
#pragma unroll
    for (int nb = 0; nb < 2; ++nb)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int i = rb * 8 + nb * 4 + c;
        float v = num[0][rb][nb][c];
        if (halves) {  // groups 0, 2 here and 1, 3 in the second half
          v += red[i * 32];
          if (A.ks_n == 4) {
            v += num[1][rb][nb][c];
            v += red[(32 + i) * 32];
          }
        } else {
#pragma unroll
          for (int q = 1; q < GN; ++q)
            if (q < A.ks_n) v += num[q][rb][nb][c];
        }
        av[nb][c] += v;
      }
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const int row = 16 * rb + g + 8 * hf, x = frame_row(A, f, row);
      const float den = den_s[row];
      if (x >= 0) {
#pragma unroll
        for (int nb = 0; nb < 2; ++nb)
          store2(og + (size_t)x * D + cb + 8 * nb + 2 * t, den != 0.f ? av[nb][2 * hf] / den : 0.f,
                 den != 0.f ? av[nb][2 * hf + 1] / den : 0.f);
      }
    }
  }
}

// ------------------------------------------------------------------ backward
// The row kernels: warp (r, h) has rows 16 r .. 16 r + 15 of the frame and the h-th
// 16 features of every staged chunk of 32; what the two halves sum over features
// is added at the end.

// Projections of 16 rows onto 16 staged features (rows f0.. of Om).
template <typename IO, int D>
__device__ __forceinline__ void project16(const bf16* Xs, int r0, const bf16* Om, int f0,
                                          float (&acc)[2][4]) {
  constexpr int NX = Pieces<IO>::NX, PD = D + 8;
  float lo[2][4] = {};
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks) {
    uint32_t a[NX][4], b[3][4];
    ld_a<NX>(a, Xs, kTile * PD, PD, r0, 16 * ks);
    ld_b<3>(b, Om, kChunk * PD, PD, f0, 16 * ks);
    mma_project<NX, 3>(acc[0], acc[1], lo[0], lo[1], a, b);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] += lo[i][c];
}

// g(X) of a frame in the backward.  FP: from FMA projections (fp32 problems with
// d <= 32, where they are the more exact and cheap); otherwise from MMAs.
template <typename IO, int D>
struct RowFeatures {
  static constexpr int NX = Pieces<IO>::NX, PD = D + 8;
  static constexpr bool FP = NX == 3 && D <= 32;
  static constexpr int kPitch = kChunk + 4;
  // shared memory of the FMA projections: rows, two chunks of Omega, a chunk of g(X)
  static constexpr int xs = FP ? kTile * fp_pitch<D>() : 0, omf = FP ? D * kChunk : 0,
                       ph = FP ? kTile * kPitch : 0, floats = xs + 2 * omf + ph;

  // this warp's 16 rows at features fg .. fg + 15 (fl: the same features' offset in
  // the chunk); x0, x1: caller rows of this thread's rows (-1: padding, g = 0)
  static __device__ __forceinline__ void get(const TileArgs& A, const IO* xg, const bf16* Xs,
                                             const float* hx, const bf16* Om, const float* phs, int r0,
                                             int fl, int fg, int x0, int x1, float (&phi)[2][4]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    if (FP) {
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const float2 v = *reinterpret_cast<const float2*>(
              phs + (r0 + g + 8 * hf) * kPitch + fl + 8 * i + 2 * t);
          phi[i][2 * hf] = v.x;
          phi[i][2 * hf + 1] = v.y;
        }
      return;
    }
    if (A.feature == SLIM_FEAT_SQUARE) {
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float x = staged<NX>(
              Xs + (r0 + g + 8 * (c >> 1)) * PD + fg + 8 * i + 2 * t + (c & 1), kTile * PD);
          phi[i][c] = x * x;
        }
      return;
    }
    project16<IO, D>(Xs, r0, Om, fl, phi);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int r = r0 + g + 8 * (c >> 1), f = fg + 8 * i + 2 * t + (c & 1), x = c >> 1 ? x1 : x0;
        phi[i][c] = x >= 0 ? feature_value<IO>(A, phi[i][c], hx[r], f, xg + (size_t)x * D, D) : 0.f;
      }
  }
};

// dOmega partials: CTA i of a backward launch adds the products of its tiles, in
// the order it takes them, onto partial i.  Partials hold the accumulators as the
// lanes do: 16 features x 16 columns are 2 x 32 float4 (slot_at), so that a warp
// moves 512 contiguous bytes; k_domega puts them back in order.
__device__ __forceinline__ size_t slot_at(int mb, int kd, int n16, int n8) {
  return ((size_t)((mb * kd + n16) * 2 + n8) * 32 + (threadIdx.x & 31)) * 4;
}
__device__ __forceinline__ void slot_put(float* p, const float (&v)[4], bool first) {
  if (first)
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v[0]),
                 "f"(v[1]), "f"(v[2]), "f"(v[3])
                 : "memory");
}
// the pieces of a 16 x 16 block (as an A fragment) to rows r0.. of a row-major
// tile, columns col0..
template <int NP>
__device__ __forceinline__ void put_block(bf16* dst, size_t ps, int pitch, int r0, int col0,
                                          const uint32_t (&a)[NP][4]) {
  const int lane = threadIdx.x & 31;
  dst += (size_t)(r0 + (lane >> 2)) * pitch + col0 + 2 * (lane & 3);
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    bf16* d = dst + p * ps;
    *reinterpret_cast<uint32_t*>(d) = a[p][0];
    *reinterpret_cast<uint32_t*>(d + (size_t)8 * pitch) = a[p][1];
    *reinterpret_cast<uint32_t*>(d + 8) = a[p][2];
    *reinterpret_cast<uint32_t*>(d + (size_t)8 * pitch + 8) = a[p][3];
  }
}
// u = dg (.) g'(x) of 16 rows x 16 features from dg and g (exp: g' = g; ReLU: 0 or
// 1 / sqrt(M)), in place
__device__ __forceinline__ void feature_vjp(const TileArgs& A, float (&dphi)[2][4],
                                            const float (&phi)[2][4]) {
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c)
      dphi[i][c] = A.feature == SLIM_FEAT_EXP ? dphi[i][c] * phi[i][c]
                                              : (phi[i][c] > 0.f ? dphi[i][c] * A.inv_sqrt_m : 0.f);
}
// quadratic map: dX = 2 x (.) dg, straight to the caller's rows
template <typename IO, int D>
__device__ __forceinline__ void store_square_vjp(IO* dst, const bf16* Xs, int r0, int fg, int x0,
                                                 int x1, const float (&dphi)[2][4]) {
  constexpr int NX = Pieces<IO>::NX, PD = D + 8;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const int row = hf ? x1 : x0, col = fg + 8 * i + 2 * t;
      const bf16* x = Xs + (r0 + g + 8 * hf) * PD + col;
      if (row >= 0)
        store2(dst + (size_t)row * D + col, 2.f * staged<NX>(x, kTile * PD) * dphi[i][2 * hf],
               2.f * staged<NX>(x + 1, kTile * PD) * dphi[i][2 * hf + 1]);
    }
}
// dX = u Omega (- x sum u for the exponential map) of 16 rows, columns in D / 8 n8 blocks
template <typename IO, int D>
__device__ __forceinline__ void store_dx(const TileArgs& A, IO* dst, const bf16* Xs, int r0, int x0,
                                         int x1, const float (&dx)[D / 8][4], float us0, float us1) {
  constexpr int NX = Pieces<IO>::NX, PD = D + 8;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const bool ex = A.feature == SLIM_FEAT_EXP;
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    const int row = hf ? x1 : x0;
    const float us = hf ? us1 : us0;
    if (row >= 0) {
#pragma unroll
      for (int i = 0; i < D / 8; ++i) {
        float x = dx[i][2 * hf], y = dx[i][2 * hf + 1];
        if (ex) {
          const bf16* xs = Xs + (r0 + g + 8 * hf) * PD + 8 * i + 2 * t;
          x -= staged<NX>(xs, kTile * PD) * us;
          y -= staged<NX>(xs + 1, kTile * PD) * us;
        }
        store2(dst + (size_t)row * D + 8 * i + 2 * t, x, y);
      }
    }
  }
}

// CTAs that fit an SM by shared memory (228 KB, 1 KB of it per CTA)
constexpr int ctas_per_sm(int bytes) { return 2 * (bytes + 1024) <= 233472 ? 2 : 1; }

constexpr int kPT = kChunk + 8;  // row pitch of the 64 x 32 chunk tiles

template <typename IO, int D>
struct BwdQSmem {
  static constexpr int NX = Pieces<IO>::NX, NS = Pieces<IO>::NS, PD = D + 8, PK = kTile + 8;
  static constexpr int X = NX * kTile * PD, W = NS * kTile * PD, OM = 3 * kChunk * PD,
                       PP = NS * kChunk * PD, KT = NS * kTile * kPT, R = OM + PP + KT,
                       TQ = NS * kTile * kPT, DA = NS * kTile * PK;
  static constexpr bool V_OWN = NX == 1;  // V has its own place, or takes the chunk's
  static constexpr int bytes = (X + W + R + 2 * TQ + DA + (V_OWN ? X : 0)) * 2 + 4 * kTile * 4 + 4 * kChunk * 4 +
                               RowFeatures<IO, D>::floats * 4;
  static_assert(V_OWN || X <= R, "V in the chunk buffers");
  static_assert(OM + KT <= 2 * TQ + DA, "second chunk buffer");
  static_assert(128 * 34 * 4 <= 2 * TQ * 2, "score sums");
  static_assert(128 * (D / 2 + 2) * 4 <= R * 2, "dq sums");
  static_assert(bytes <= kSmemMax, "shared memory");
};
template <typename IO, int D>
struct BwdKSmem {
  static constexpr int NX = Pieces<IO>::NX, NS = Pieces<IO>::NS, PD = D + 8, PK = kTile + 8;
  static constexpr int X = NX * kTile * PD, OM = 3 * kChunk * PD, GG = NS * kChunk * PD,
                       TQ = NS * kTile * kPT, DA = NS * kTile * PK, W = NS * kTile * PD,
                       R = OM + GG + 2 * TQ + DA;
  static constexpr int bytes = (2 * X + R) * 2 + kTile * 4 + RowFeatures<IO, D>::floats * 4;
  static_assert(DA + W <= R, "A and dnum in the chunk buffers");
  static_assert(128 * (D + 2) * 4 <= R * 2, "dk, dv sums");
  static_assert(bytes <= kSmemMax, "shared memory");
};
template <typename IO, int D>
constexpr int bwd_occupancy() {
  return ctas_per_sm(BwdQSmem<IO, D>::bytes) == 2 && ctas_per_sm(BwdKSmem<IO, D>::bytes) == 2 ? 2 : 1;
}

// Query side of a tile, from its state P_t:
//   den = g(Q) z + A 1, dnum = dout / den, dden = -<dout, out> / den,
//   dA = tril(dnum V^T + dden), dg(Q) = dnum S^T + dden z + dA g(K),
//   Gd = g(Q)^T [dnum | dden], u = dg(Q) (.) g'(q), dq = u Omega - q sum u, dOmega += u^T q.
// Two passes over the features: the first sums the denominators and A, which the
// second needs.  g(Q), A, dA and dnum are left (as pieces) for the key side.
// Bound by the dependent chain and the instructions of each product: issue 20 %, tensor
// pipe 27 %, 8 warps on an SM in fp32 (158 KB, 255 registers); 768 frames of d = 64, M = 128
// take 272 us (k_bwd_k 169 us).  Sixteen warps and half the features each: 1.5 times the
// instructions, 2.6 % slower.
template <typename IO, int D>
__global__ void __launch_bounds__(kThreads, (bwd_occupancy<IO, D>()))
    k_bwd_q(const __grid_constant__ TileArgs A) {
  using S = BwdQSmem<IO, D>;
  constexpr int NX = S::NX, NS = S::NS, PD = S::PD, PK = S::PK, KD = D / 16;
  extern __shared__ uint4 smem_raw[];
  bf16* Xs = reinterpret_cast<bf16*>(smem_raw);
  bf16* Ws = Xs + S::X;
  bf16* Om = Ws + S::W;
  bf16* Ps = Om + S::OM;
  bf16* Kt = Ps + S::PP;
  bf16* Tq = Kt + S::KT;
  bf16* Tu = Tq + S::TQ;
  bf16* dAs = Tu + S::TQ;
  bf16* Vs = S::V_OWN ? dAs + S::DA : Om;
  float* hx = reinterpret_cast<float*>(dAs + S::DA + (S::V_OWN ? S::X : 0));
  float* rd = hx + kTile;   // <dout, out>, then dden
  float* dn = rd + kTile;   // den
  float* gzs = dn + 2 * kTile;  // [4][kChunk]
  using F = RowFeatures<IO, D>;
  float* xf = gzs + 4 * kChunk;  // FMA projections
  float* omf = xf + F::xs;
  float* phs = omf + 2 * F::omf;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, g = lane >> 2, t = lane & 3;
  const int h = warp >> 2, rb = warp & 3, r0 = 16 * rb, fl = 16 * h;
  const bool square = A.feature == SLIM_FEAT_SQUARE;
  const size_t MD = (size_t)A.M * D;
  float* slot = A.slots + (size_t)blockIdx.x * MD;

  for (int tile = blockIdx.x; tile < A.chains * A.nf; tile += gridDim.x) {
    const Frame tp = frame_pos(A, tile);
    const bool first = tile == (int)blockIdx.x;
    const int x0 = frame_row(A, tp, r0 + g), x1 = frame_row(A, tp, r0 + g + 8);
    const IO* qg = static_cast<const IO*>(A.q) + tp.row0 * D;
    const IO* vg = static_cast<const IO*>(A.v) + tp.row0 * D;
    const IO* dog = static_cast<const IO*>(A.dout) + tp.row0 * D;
    const IO* og = static_cast<const IO*>(A.out) + tp.row0 * D;
    const float* Pt = A.P + tp.c * A.p_chain + tp.t0 / A.per * A.p_frame;
    const bf16* kt = A.phi_k + (size_t)tile * NS * A.M * kTile;
    bf16* pq = A.phi_q + (size_t)tile * NS * A.M * kTile;
    bf16* sA = A.sA + (size_t)tile * NS * kTile * kTile;
    bf16* sdA = A.sdA + (size_t)tile * NS * kTile * kTile;
    bf16* sW = A.sW + (size_t)tile * NS * kTile * D;
    float* gd = A.gdelta + (size_t)tile * A.E;

    auto stage = [&](int c0, bf16* om, bf16* ktp, float* of) {
      const int nf = min(kChunk, A.M - c0);
      if (!square)
        stage_rows<3>(om, kChunk * PD, PD, A.om_row + (size_t)c0 * D, MD, D, nf, D);
      if (A.causal)
        stage_rows<NS>(ktp, kTile * kPT, kPT, kt + c0, (size_t)A.M * kTile, A.M, kTile, nf);
      if (F::FP && !square) stage_omega<D, kChunk>(of, A.om_t, c0);
      cp_commit();
    };
    // g(Q) of a chunk by FMAs (ends with a barrier)
    auto project_fp = [&](int c0, const float* of) {
      features_fp<D, kChunk>(A, tp, xf, dn + kTile, of, c0,
                             [&](int r, int fo, const float(&v)[2]) {
                               *reinterpret_cast<float2*>(phs + r * F::kPitch + fo) = make_float2(v[0], v[1]);
                             });
      __syncthreads();
    };
    // pass 1's chunks alternate between the chunk buffers and the T | dA space
    bf16* om2 = Tq;
    bf16* kt2 = Tq + S::OM;
    stage(0, Om, Kt, omf);
    load_rows<IO, D>(A, tp, qg, Xs, hx);
    if (F::FP) load_rows_fp<IO, D>(A, tp, qg, xf);
    if (S::V_OWN) load_rows<IO, D>(A, tp, vg, Vs, nullptr);
    for (int e = tid; e < kTile * (D / 8); e += kThreads) {
      const int r = e / (D / 8), c8 = (e % (D / 8)) * 8;
      const int x = frame_row(A, tp, r);
      float s = 0.f;
      if (x >= 0) {
        float a[8], b[8];
        load8(dog + (size_t)x * D + c8, a);
        load8(og + (size_t)x * D + c8, b);
#pragma unroll
        for (int i = 0; i < 8; ++i) s = fmaf(a[i], b[i], s);
      }
#pragma unroll
      for (int o = 1; o < D / 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (c8 == 0) rd[r] = s;
    }
    cp_wait<0>();
    __syncthreads();
    if (F::FP) {
      row_norms<D>(xf, dn + kTile);
      __syncthreads();
    }
    pdl_wait();  // the state; all staged so far is older (a no-op after the first frame)
    pdl_launch();

    // pass 1: g(Q), A, den
    float den0 = 0.f, den1 = 0.f;
    {
      float sc[8][4] = {};
      int cur = 0;
      for (int c0 = 0; c0 < A.M; c0 += kChunk) {
        if (c0 + kChunk < A.M) stage(c0 + kChunk, cur ? Om : om2, cur ? Kt : kt2, cur ? omf : omf + F::omf);
        const bf16* om = cur ? om2 : Om;
        const bf16* ktp = cur ? kt2 : Kt;
        if (F::FP) project_fp(c0, cur ? omf + F::omf : omf);
        const int fg = c0 + fl;
        if (fg < A.M) {
          float phi[2][4];
          F::get(A, qg, Xs, hx, om, phs, r0, fl, fg, x0, x1, phi);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float2 z = *reinterpret_cast<const float2*>(Pt + MD + fg + 8 * i + 2 * t);
            den0 = fmaf(phi[i][0], z.x, fmaf(phi[i][1], z.y, den0));
            den1 = fmaf(phi[i][2], z.x, fmaf(phi[i][3], z.y, den1));
          }
          if (A.causal) {
            uint32_t a[NS][4];
            acc_to_a<NS>(a, phi[0], phi[1]);
            put_block<NS>(pq, (size_t)kTile * A.M, A.M, r0, fg, a);
#pragma unroll
            for (int kb = 0; kb < 4; ++kb)
              if (kb <= rb) {
                uint32_t b[NS][4];
                ld_b<NS>(b, ktp, kTile * kPT, kPT, 16 * kb, fl);
                mma_sum<NS, NS>(sc[2 * kb], sc[2 * kb + 1], a, b);
              }
          }
        }
        cp_wait<0>();
        __syncthreads();
        cur ^= 1;
      }
      den0 = quad_sum(den0);
      den1 = quad_sum(den1);
      float* red = reinterpret_cast<float*>(Tq) + (tid & 127);
      if (h == 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) red[(4 * i + c) * 128] = sc[i][c];
        red[32 * 128] = den0;
        red[33 * 128] = den1;
      }
      __syncthreads();
      if (S::V_OWN) {  // the chunk buffers are free: pass 2's first chunk
        stage(0, Om, Kt, omf);
      } else {
        load_rows<IO, D>(A, tp, vg, Vs, nullptr);
      }
      if (h == 0) {
        den0 += red[32 * 128];
        den1 += red[33 * 128];
        if (A.causal) {
          float a0 = 0.f, a1 = 0.f;
#pragma unroll
          for (int kb = 0; kb < 4; ++kb)
            if (kb <= rb) {
#pragma unroll
              for (int i = 2 * kb; i < 2 * kb + 2; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  const int row = r0 + g + 8 * (c >> 1), key = 8 * i + 2 * t + (c & 1);
                  const float v = sc[i][c] + red[(4 * i + c) * 128];
                  sc[i][c] = key <= row ? v : 0.f;
                }
              a0 += sc[2 * kb][0] + sc[2 * kb][1] + sc[2 * kb + 1][0] + sc[2 * kb + 1][1];
              a1 += sc[2 * kb][2] + sc[2 * kb][3] + sc[2 * kb + 1][2] + sc[2 * kb + 1][3];
              uint32_t a[NS][4];
              acc_to_a<NS>(a, sc[2 * kb], sc[2 * kb + 1]);
              put_block<NS>(sA, kTile * kTile, kTile, r0, 16 * kb, a);
            }
          den0 += quad_sum(a0);
          den1 += quad_sum(a1);
        }
        if (t == 0) {
          dn[r0 + g] = den0;
          dn[r0 + g + 8] = den1;
        }
      }
    }
    __syncthreads();

    // W = dnum (pieces), dden
    for (int e = tid; e < kTile * (D / 8); e += kThreads) {
      const int r = e / (D / 8), c8 = (e % (D / 8)) * 8;
      const int x = frame_row(A, tp, r);
      const float den = dn[r];
      float v[8] = {};
      if (x >= 0 && den != 0.f) {
        load8(dog + (size_t)x * D + c8, v);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = v[i] / den;
      }
      store_pieces8<NS>(Ws + r * PD + c8, kTile * PD, v);
      if (A.causal) store_pieces8<NS>(sW + r * D + c8, kTile * D, v);
    }
    if (tid < kTile) {
      const float den = dn[tid];
      rd[tid] = frame_row(A, tp, tid) >= 0 && den != 0.f ? -rd[tid] / den : 0.f;
    }
    __syncthreads();
    const float dd0 = rd[r0 + g], dd1 = rd[r0 + g + 8];

    if (A.causal) {  // dA, a half's warp taking every other block of 16 keys
#pragma unroll
      for (int kb = 0; kb < 4; ++kb)
        if (kb <= rb && (kb & 1) == h) {
          float d[2][4] = {};
#pragma unroll
          for (int ks = 0; ks < KD; ++ks) {
            uint32_t a[NS][4], b[NX][4];
            ld_a<NS>(a, Ws, kTile * PD, PD, r0, 16 * ks);
            ld_b<NX>(b, Vs, kTile * PD, PD, 16 * kb, 16 * ks);
            mma_sum<NS, NX>(d[0], d[1], a, b);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const int row = r0 + g + 8 * (c >> 1), key = 16 * kb + 8 * i + 2 * t + (c & 1);
              d[i][c] = key <= row ? d[i][c] + (c >> 1 ? dd1 : dd0) : 0.f;
            }
          uint32_t a[NS][4];
          acc_to_a<NS>(a, d[0], d[1]);
          put_block<NS>(dAs, kTile * PK, PK, r0, 16 * kb, a);
          put_block<NS>(sdA, kTile * kTile, kTile, r0, 16 * kb, a);
        }
    }
    StateChunk<D, kChunk> pc;
    if (!S::V_OWN) {
      __syncthreads();  // V read: the chunk buffers are free
      stage(0, Om, Kt, omf);
    }
    pc.load(Pt, min(kChunk, A.M));
    pc.template store<NS>(Ps, min(kChunk, A.M));
    cp_wait<0>();
    __syncthreads();

    // pass 2
    float dq[D / 8][4] = {}, us0 = 0.f, us1 = 0.f;
    for (int c0 = 0; c0 < A.M; c0 += kChunk) {
      const int fg = c0 + fl;
      if (F::FP) project_fp(c0, omf);
      if (fg < A.M) {
        float phi[2][4], dp[2][4] = {};
        F::get(A, qg, Xs, hx, Om, phs, r0, fl, fg, x0, x1, phi);
#pragma unroll
        for (int ks = 0; ks < KD; ++ks) {
          uint32_t a[NS][4], b[NS][4];
          ld_a<NS>(a, Ws, kTile * PD, PD, r0, 16 * ks);
          ld_b<NS>(b, Ps, kChunk * PD, PD, fl, 16 * ks);
          mma_sum<NS, NS>(dp[0], dp[1], a, b);
        }
        if (A.causal) {
#pragma unroll
          for (int kb = 0; kb < 4; ++kb)
            if (kb <= rb) {
              uint32_t a[NS][4], b[NS][4];
              ld_a<NS>(a, dAs, kTile * PK, PK, r0, 16 * kb);
              ld_bt<NS>(b, Kt, kTile * kPT, kPT, fl, 16 * kb);
              mma_sum<NS, NS>(dp[0], dp[1], a, b);
            }
        }
        uint32_t a[NS][4];
        acc_to_a<NS>(a, phi[0], phi[1]);
        put_block<NS>(Tq, kTile * kPT, kPT, r0, fl, a);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float2 z = *reinterpret_cast<const float2*>(Pt + MD + fg + 8 * i + 2 * t);
          dp[i][0] = fmaf(dd0, z.x, dp[i][0]);
          dp[i][1] = fmaf(dd0, z.y, dp[i][1]);
          dp[i][2] = fmaf(dd1, z.x, dp[i][2]);
          dp[i][3] = fmaf(dd1, z.y, dp[i][3]);
          // g_z's share: sum over this warp's rows of g(Q) dden
          float s0 = fmaf(phi[i][0], dd0, phi[i][2] * dd1), s1 = fmaf(phi[i][1], dd0, phi[i][3] * dd1);
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
          }
          if (g == 0) {
            gzs[rb * kChunk + fl + 8 * i + 2 * t] = s0;
            gzs[rb * kChunk + fl + 8 * i + 2 * t + 1] = s1;
          }
        }
        if (square) {
          store_square_vjp<IO, D>(static_cast<IO*>(A.dq) + tp.row0 * D, Xs, r0, fg, x0, x1, dp);
        } else {
          feature_vjp(A, dp, phi);
          us0 += dp[0][0] + dp[0][1] + dp[1][0] + dp[1][1];
          us1 += dp[0][2] + dp[0][3] + dp[1][2] + dp[1][3];
          acc_to_a<NS>(a, dp[0], dp[1]);
          put_block<NS>(Tu, kTile * kPT, kPT, r0, fl, a);
#pragma unroll
          for (int nb = 0; nb < KD; ++nb) {
            uint32_t b[NS][4];
            ld_bt<NS>(b, Om, kChunk * PD, PD, 16 * nb, fl);
            mma_sum<NS, NS>(dq[2 * nb], dq[2 * nb + 1], a, b);
          }
        }
      }
      __syncthreads();
      const bool more = c0 + kChunk < A.M;
      if (more) {
        stage(c0 + kChunk, Om, Kt, omf);
        pc.load(Pt + (size_t)(c0 + kChunk) * D, min(kChunk, A.M - c0 - kChunk));
      }
      // warps 0-3: Gd = g(Q)^T dnum; warps 4-7: dOmega += u^T q; each 16 features x
      // half of the columns (all of them for d = 16)
      const int mb = (warp >> 1) & 1, ng = warp & 1;
      constexpr int NU = KD >= 2 ? KD / 2 : 1;
      if (c0 + 16 * mb < A.M && (KD >= 2 || ng == 0) && (h == 0 || !square)) {
        float o[2 * NU][4] = {};
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          uint32_t a[NS][4];
          ld_at<NS>(a, h ? Tu : Tq, kTile * kPT, kPT, 16 * mb, 16 * ks);
#pragma unroll
          for (int nu = 0; nu < NU; ++nu) {
            const int n0 = 16 * (ng * NU + nu);
            if (h == 0) {
              uint32_t b[NS][4];
              ld_bt<NS>(b, Ws, kTile * PD, PD, n0, 16 * ks);
              mma_sum<NS, NS>(o[2 * nu], o[2 * nu + 1], a, b);
            } else {
              uint32_t b[NX][4];
              ld_bt<NX>(b, Xs, kTile * PD, PD, n0, 16 * ks);
              mma_sum<NS, NX>(o[2 * nu], o[2 * nu + 1], a, b);
            }
          }
        }
#pragma unroll
        for (int nu = 0; nu < NU; ++nu)
#pragma unroll
          for (int n8 = 0; n8 < 2; ++n8) {
            const float(&v)[4] = o[2 * nu + n8];
            if (h == 0) {
              float* dst = gd + (size_t)(c0 + 16 * mb + g) * D + 16 * (ng * NU + nu) + 8 * n8 + 2 * t;
              *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
              *reinterpret_cast<float2*>(dst + 8 * D) = make_float2(v[2], v[3]);
            } else {
              slot_put(slot + slot_at(c0 / 16 + mb, KD, ng * NU + nu, n8), v, first);
            }
          }
      }
      if (tid < kChunk && c0 + tid < A.M)
        gd[MD + c0 + tid] = (gzs[tid] + gzs[kChunk + tid]) + (gzs[2 * kChunk + tid] + gzs[3 * kChunk + tid]);
      if (more) pc.template store<NS>(Ps, min(kChunk, A.M - c0 - kChunk));
      cp_wait<0>();
      __syncthreads();
    }
    if (!square) {
      us0 = quad_sum(us0);
      us1 = quad_sum(us1);
      float* red = reinterpret_cast<float*>(Om) + (tid & 127);
      if (h == 1) {
#pragma unroll
        for (int i = 0; i < D / 8; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) red[(4 * i + c) * 128] = dq[i][c];
        red[(D / 2) * 128] = us0;
        red[(D / 2 + 1) * 128] = us1;
      }
      __syncthreads();
      if (h == 0) {
#pragma unroll
        for (int i = 0; i < D / 8; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) dq[i][c] += red[(4 * i + c) * 128];
        store_dx<IO, D>(A, static_cast<IO*>(A.dq) + tp.row0 * D, Xs, r0, x0, x1, dq,
                        us0 + red[(D / 2) * 128], us1 + red[(D / 2 + 1) * 128]);
      }
    }
    __syncthreads();  // before the next tile's loads
  }
}

// Key / value side of a tile, from its state gradient G_t and the query side's
// g(Q), A, dA and dnum:
//   dg(K) = V G_S^T + g_z + dA^T g(Q), dV = g(K) G_S + A^T dnum,
//   u = dg(K) (.) g'(k), dk = u Omega - k sum u, dOmega += u^T k.
template <typename IO, int D>
__global__ void __launch_bounds__(kThreads, (bwd_occupancy<IO, D>()))
    k_bwd_k(const __grid_constant__ TileArgs A) {
  using S = BwdKSmem<IO, D>;
  constexpr int NX = S::NX, NS = S::NS, PD = S::PD, PK = S::PK, KD = D / 16;
  extern __shared__ uint4 smem_raw[];
  bf16* Ks = reinterpret_cast<bf16*>(smem_raw);
  bf16* Vs = Ks + S::X;
  bf16* Om = Vs + S::X;
  bf16* Gs = Om + S::OM;
  bf16* Qs = Gs + S::GG;
  bf16* Tu = Qs + S::TQ;
  bf16* dAs = Tu + S::TQ;
  float* hx = reinterpret_cast<float*>(dAs + S::DA);
  using F = RowFeatures<IO, D>;
  float* xf = hx + kTile;  // FMA projections (one chunk of Omega; the other's space holds |x|^2)
  float* omf = xf + F::xs;
  float* norm2 = omf + F::omf;
  float* phs = omf + 2 * F::omf;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, g = lane >> 2, t = lane & 3;
  const int h = warp >> 2, rb = warp & 3, r0 = 16 * rb, fl = 16 * h;
  const bool square = A.feature == SLIM_FEAT_SQUARE;
  const size_t MD = (size_t)A.M * D;
  float* slot = A.slots + (size_t)blockIdx.x * MD;

  for (int tile = blockIdx.x; tile < A.chains * A.nf; tile += gridDim.x) {
    const Frame tp = frame_pos(A, tile);
    const int x0 = frame_row(A, tp, r0 + g), x1 = frame_row(A, tp, r0 + g + 8);
    const IO* kg = static_cast<const IO*>(A.k) + tp.row0 * D;
    const float* Gt = A.G + tp.c * A.g_chain + tp.t0 / A.per * A.g_frame;
    const bf16* pq = A.phi_q + (size_t)tile * NS * A.M * kTile;
    const bf16* sA = A.sA + (size_t)tile * NS * kTile * kTile;
    const bf16* sdA = A.sdA + (size_t)tile * NS * kTile * kTile;
    const bf16* sW = A.sW + (size_t)tile * NS * kTile * D;

    StateChunk<D, kChunk> gc;
    auto stage = [&](int c0) {
      const int nf = min(kChunk, A.M - c0);
      if (!square)
        stage_rows<3>(Om, kChunk * PD, PD, A.om_row + (size_t)c0 * D, MD, D, nf, D);
      if (A.causal)
        stage_rows<NS>(Qs, kTile * kPT, kPT, pq + c0, (size_t)kTile * A.M, A.M, kTile, nf);
      if (F::FP && !square) stage_omega<D, kChunk>(omf, A.om_t, c0);
      cp_commit();
    };
    if (A.causal) stage_rows<NS>(dAs, kTile * PK, PK, sdA, kTile * kTile, kTile, kTile, kTile);
    stage(0);
    load_rows<IO, D>(A, tp, kg, Ks, hx);
    if (F::FP) load_rows_fp<IO, D>(A, tp, kg, xf);
    load_rows<IO, D>(A, tp, static_cast<const IO*>(A.v) + tp.row0 * D, Vs, nullptr);
    pdl_wait();  // the state gradient; all staged so far is older
    pdl_launch();
    gc.load(Gt, min(kChunk, A.M));
    gc.template store<NS>(Gs, min(kChunk, A.M));
    cp_wait<0>();
    __syncthreads();
    if (F::FP) {
      row_norms<D>(xf, norm2);
      __syncthreads();
    }

    float dk[D / 8][4] = {}, dv[D / 8][4] = {}, us0 = 0.f, us1 = 0.f;
    for (int c0 = 0; c0 < A.M; c0 += kChunk) {
      const int fg = c0 + fl;
      if (F::FP) {
        features_fp<D, kChunk>(A, tp, xf, norm2, omf, c0, [&](int r, int fo, const float(&v)[2]) {
          *reinterpret_cast<float2*>(phs + r * F::kPitch + fo) = make_float2(v[0], v[1]);
        });
        __syncthreads();
      }
      if (fg < A.M) {
        float phi[2][4], dp[2][4] = {};
        F::get(A, kg, Ks, hx, Om, phs, r0, fl, fg, x0, x1, phi);
#pragma unroll
        for (int ks = 0; ks < KD; ++ks) {
          uint32_t a[NX][4], b[NS][4];
          ld_a<NX>(a, Vs, kTile * PD, PD, r0, 16 * ks);
          ld_b<NS>(b, Gs, kChunk * PD, PD, fl, 16 * ks);
          mma_sum<NX, NS>(dp[0], dp[1], a, b);
        }
        if (A.causal) {
#pragma unroll
          for (int kb = 0; kb < 4; ++kb)
            if (kb >= rb) {  // rows before these keys do not read them
              uint32_t a[NS][4], b[NS][4];
              ld_at<NS>(a, dAs, kTile * PK, PK, r0, 16 * kb);
              ld_bt<NS>(b, Qs, kTile * kPT, kPT, fl, 16 * kb);
              mma_sum<NS, NS>(dp[0], dp[1], a, b);
            }
        }
        uint32_t a[NS][4];
        acc_to_a<NS>(a, phi[0], phi[1]);
#pragma unroll
        for (int nb = 0; nb < KD; ++nb) {
          uint32_t b[NS][4];
          ld_bt<NS>(b, Gs, kChunk * PD, PD, 16 * nb, fl);
          mma_sum<NS, NS>(dv[2 * nb], dv[2 * nb + 1], a, b);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float2 z = *reinterpret_cast<const float2*>(Gt + MD + fg + 8 * i + 2 * t);
          dp[i][0] += z.x;
          dp[i][1] += z.y;
          dp[i][2] += z.x;
          dp[i][3] += z.y;
        }
        if (square) {
          store_square_vjp<IO, D>(static_cast<IO*>(A.dk) + tp.row0 * D, Ks, r0, fg, x0, x1, dp);
        } else {
          feature_vjp(A, dp, phi);
          us0 += dp[0][0] + dp[0][1] + dp[1][0] + dp[1][1];
          us1 += dp[0][2] + dp[0][3] + dp[1][2] + dp[1][3];
          acc_to_a<NS>(a, dp[0], dp[1]);
          put_block<NS>(Tu, kTile * kPT, kPT, r0, fl, a);
#pragma unroll
          for (int nb = 0; nb < KD; ++nb) {
            uint32_t b[NS][4];
            ld_bt<NS>(b, Om, kChunk * PD, PD, 16 * nb, fl);
            mma_sum<NS, NS>(dk[2 * nb], dk[2 * nb + 1], a, b);
          }
        }
      }
      __syncthreads();
      const bool more = c0 + kChunk < A.M;
      if (more) {
        stage(c0 + kChunk);
        gc.load(Gt + (size_t)(c0 + kChunk) * D, min(kChunk, A.M - c0 - kChunk));
      }
      if (!square) {
        for (int u = warp; u < 2 * KD; u += kThreads / 32) {  // 16 features x 16 columns
          const int mb = u & 1, n16 = u >> 1;
          if (c0 + 16 * mb < A.M) {
            float o[2][4] = {};
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
              uint32_t a[NS][4], b[NX][4];
              ld_at<NS>(a, Tu, kTile * kPT, kPT, 16 * mb, 16 * ks);
              ld_bt<NX>(b, Ks, kTile * PD, PD, 16 * n16, 16 * ks);
              mma_sum<NS, NX>(o[0], o[1], a, b);
            }
#pragma unroll
            for (int n8 = 0; n8 < 2; ++n8)
              slot_put(slot + slot_at(c0 / 16 + mb, KD, n16, n8), o[n8],
                       A.slots_new && tile == (int)blockIdx.x);
          }
        }
      }
      if (more) gc.template store<NS>(Gs, min(kChunk, A.M - c0 - kChunk));
      cp_wait<0>();
      __syncthreads();
    }
    if (A.causal) {  // dV += A^T dnum, a half's warps taking every other block of 16 rows
      bf16* As = Om;
      bf16* Ws = Om + S::DA;
      stage_rows<NS>(As, kTile * PK, PK, sA, kTile * kTile, kTile, kTile, kTile);
      stage_rows<NS>(Ws, kTile * PD, PD, sW, kTile * D, D, kTile, D);
      cp_commit();
      cp_wait<0>();
      __syncthreads();
#pragma unroll
      for (int kb = 0; kb < 4; ++kb)
        if (kb >= rb && (kb & 1) == h) {
          uint32_t a[NS][4];
          ld_at<NS>(a, As, kTile * PK, PK, r0, 16 * kb);
#pragma unroll
          for (int nb = 0; nb < KD; ++nb) {
            uint32_t b[NS][4];
            ld_bt<NS>(b, Ws, kTile * PD, PD, 16 * nb, 16 * kb);
            mma_sum<NS, NS>(dv[2 * nb], dv[2 * nb + 1], a, b);
          }
        }
      __syncthreads();
    }
    // half 0 finishes dk, half 1 dv, each with the other's sums
    us0 = quad_sum(us0);
    us1 = quad_sum(us1);
    float* rk = reinterpret_cast<float*>(Om) + (tid & 127);
    float* rv = rk + (D / 2 + 2) * 128;
#pragma unroll
    for (int i = 0; i < D / 8; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (h == 1)
          rk[(4 * i + c) * 128] = dk[i][c];
        else
          rv[(4 * i + c) * 128] = dv[i][c];
      }
    if (h == 1) {
      rk[(D / 2) * 128] = us0;
      rk[(D / 2 + 1) * 128] = us1;
    }
    __syncthreads();
    if (h == 0) {
      if (!square) {
#pragma unroll
        for (int i = 0; i < D / 8; ++i)
#pragma unroll
          for (int c = 0; c < 4; ++c) dk[i][c] += rk[(4 * i + c) * 128];
        store_dx<IO, D>(A, static_cast<IO*>(A.dk) + tp.row0 * D, Ks, r0, x0, x1, dk,
                        us0 + rk[(D / 2) * 128], us1 + rk[(D / 2 + 1) * 128]);
      }
    } else {
      IO* dvg = static_cast<IO*>(A.dv) + tp.row0 * D;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int row = hf ? x1 : x0;
        if (row >= 0) {
#pragma unroll
          for (int i = 0; i < D / 8; ++i)
            store2(dvg + (size_t)row * D + 8 * i + 2 * t, dv[i][2 * hf] + rv[(4 * i + 2 * hf) * 128],
                   dv[i][2 * hf + 1] + rv[(4 * i + 2 * hf + 1) * 128]);
        }
      }
    }
    __syncthreads();  // before the next tile's loads
  }
}

// ------------------------------------------------------------------ launches
// One-time, per-device shared-memory limit of a kernel.
template <typename IO, int D, int K>
cudaError_t smem_limit(const void* kern, int bytes) {
  static bool set_flags[kMaxDevices] = {};
  bool* set = device_flag(set_flags);
  if (set == nullptr) return cudaErrorInvalidDevice;
  if (*set) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) *set = true;
  return e;
}

template <typename IO, int D>
cudaError_t run_delta(const TileArgs& A, cudaStream_t s) {
  constexpr int smem = DeltaSmem<IO, D>::bytes;
  cudaError_t e = smem_limit<IO, D, 0>((const void*)k_delta<IO, D>, smem);
  if (e != cudaSuccess) return e;
  const double rows = (double)A.chains * A.b;
  const double proj = A.feature == SLIM_FEAT_SQUARE ? 0.0 : 2.0;
  prof::Scope ps(prof::K_TILE_DELTA, s, (2.0 + proj) * rows * D * A.M, 2.0 * rows * D * sizeof(IO));
  // Few frames leave SMs idle: their chunks of 64 features, which share nothing but the
  // rows, then go to as many CTAs as the chip has room for (one frame of d = 128, M = 256 in
  // fp32: 47 -> 18 us; 64 frames 55 -> 36).  A frame that has an SM to itself loads its rows once.
  const unsigned frames = (unsigned)(A.chains * A.nf), chunks = (A.M + 63) / 64,
                 room = kSms * DeltaSmem<IO, D>::ctas / frames;
  const dim3 grid(frames, room < 2 ? 1 : room < chunks ? room : chunks);
  return launch_pdl(k_delta<IO, D>, grid, kThreads, smem, s, A);
}
template <typename IO, int D, int MODE, bool CAUSAL>
cudaError_t run_out_short(const TileArgs& A, cudaStream_t s) {
  constexpr int smem = ShortSmemOut<IO, D, CAUSAL>::bytes;
  cudaError_t e = smem_limit<IO, D, 2 + 2 * MODE + CAUSAL>((const void*)k_out_short<IO, D, MODE, CAUSAL>, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_out_short<IO, D, MODE, CAUSAL>, (unsigned)(A.chains * A.nf), kThreads, smem, s, A);
}
template <typename IO, int D>
cudaError_t run_out(const TileArgs& A, cudaStream_t s) {
  const double rows = (double)A.chains * A.b;
  const double proj = A.feature == SLIM_FEAT_SQUARE ? 0.0 : 2.0;
  prof::Scope ps(prof::K_TILE_OUT, s, (2.0 + proj) * rows * D * A.M,
                 (A.causal ? 3.0 : 2.0) * rows * D * sizeof(IO));
  if (A.rows == 16) return A.causal ? run_out_short<IO, D, 2, true>(A, s) : run_out_short<IO, D, 2, false>(A, s);
  if (A.rows == 32) return A.causal ? run_out_short<IO, D, 1, true>(A, s) : run_out_short<IO, D, 1, false>(A, s);
  constexpr int smem = OutSmem<IO, D>::bytes;
  cudaError_t e = smem_limit<IO, D, 1>((const void*)k_out<IO, D>, smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_out<IO, D>, (unsigned)(A.chains * A.nf), kThreads, smem, s, A);
}
template <typename IO, int D>
constexpr int slot_count() {
  return kSms * bwd_occupancy<IO, D>();
}
template <typename IO, int D>
unsigned bwd_grid(const TileArgs& A) {
  const long long tiles = (long long)A.chains * A.nf;
  return (unsigned)(tiles < slot_count<IO, D>() ? tiles : slot_count<IO, D>());
}
template <typename IO, int D>
cudaError_t run_bwd_q(const TileArgs& A, cudaStream_t s) {
  constexpr int smem = BwdQSmem<IO, D>::bytes;
  cudaError_t e = smem_limit<IO, D, 2>((const void*)k_bwd_q<IO, D>, smem);
  if (e != cudaSuccess) return e;
  const double rows = (double)A.chains * A.b;
  const double proj = A.feature == SLIM_FEAT_SQUARE ? 0.0 : 6.0;  // g(Q), dq, dOmega
  prof::Scope ps(prof::K_TILE_BWD_Q, s, (4.0 + proj) * rows * D * A.M, 5.0 * rows * D * sizeof(IO));
  return launch_pdl(k_bwd_q<IO, D>, bwd_grid<IO, D>(A), kThreads, smem, s, A);
}
template <typename IO, int D>
cudaError_t run_bwd_k(const TileArgs& A, cudaStream_t s) {
  constexpr int smem = BwdKSmem<IO, D>::bytes;
  cudaError_t e = smem_limit<IO, D, 3>((const void*)k_bwd_k<IO, D>, smem);
  if (e != cudaSuccess) return e;
  const double rows = (double)A.chains * A.b;
  const double proj = A.feature == SLIM_FEAT_SQUARE ? 0.0 : 4.0;  // dk, dOmega
  prof::Scope ps(prof::K_TILE_BWD_K, s, (4.0 + proj) * rows * D * A.M, 4.0 * rows * D * sizeof(IO));
  return launch_pdl(k_bwd_k<IO, D>, bwd_grid<IO, D>(A), kThreads, smem, s, A);
}

template <typename IO, int D>
constexpr TileKernels tile_set() {
  return TileKernels{run_delta<IO, D>, run_out<IO, D>, run_bwd_q<IO, D>, run_bwd_k<IO, D>,
                     slot_count<IO, D>()};
}

}  // namespace simt
}  // namespace slim
