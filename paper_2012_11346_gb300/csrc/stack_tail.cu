// Backward of one bf16 slice of fewer than 64 rows in the layer stack, d = 64 and M 128 or
// 256: the last slice of a stack on the tensor-core path where C does not divide L, and
// every slice where C < 64.
//
// A layer's dq, dk and dv are rounded to bf16 and feed the layers below, so in a
// stack the summation order of one short slice decides roundings that move every
// lower layer's fp32 dOmega by 1e-3 (within its distance from exact arithmetic, 1e-2,
// but far above fp32).  This kernel therefore keeps one fixed order: whole-slice
// contractions C = A B on operands in two bf16 pieces, k16 steps in order inside
// groups() interleaved groups, group sums in order, and a 65th column in fp32 FMA.
// The tile kernels (simt_tiles.cuh), which sum otherwise, serve every other call.
//
// One CTA per chain, two on an SM, every intermediate in L2 (310 or 510 KB a chain); one
// launch and the sum of the chains' dOmega, where the same contractions took 33 launches.
// Bound by the latency of its loads, element by element.  The backward of a one-layer stack
// of one slice, 33 launches against this kernel: 63 rows of 64 chains, M = 256, 620 -> 541
// us; of 512 chains 1993 -> 1795; 16 rows of 64 chains 448 -> 274 (with one block of columns per
// fragment of A 640, 2130 and 287).
#include <math.h>

#include "profiler.h"
#include "stack_tail.h"
#include "warp_mma.cuh"

namespace slim {
namespace tail {
namespace {

using namespace simt;

constexpr int D = 64, DP = D + 1, NT = 512;

struct Args {
  const __nv_bfloat16 *q, *k, *v, *out, *dout;
  const float* omega;
  StateIn st;
  GradIO gio;
  __nv_bfloat16 *dq, *dk, *dv;
  float *scratch, *part;  // per chain: the intermediates, the dOmega partial
  size_t chain;           // floats of scratch per chain
  int* err;
  int b, T, M, feature;   // rows, rows padded to 16
  float inv_sqrt_m;
};

struct Mat {  // element (i, k) at p + i rs + k cs
  float* p;
  int rs, cs;
};

// interleaved groups of a product's k16 steps
__device__ __forceinline__ int groups(int m, int n, int k) {
  const int want = n <= 16 ? 8 : m <= 16 ? 4 : m <= 32 ? 2 : 1;
  return k >= 32 * want ? want : 1;
}
// x rounded to its two pieces
__device__ __forceinline__ float pieces(float x) {
  const float h = __bfloat162float(__float2bfloat16_rn(x));
  return __bfloat162float(__float2bfloat16_rn(__fsub_rn(x, h))) + h;
}

// C = A B, a warp taking 16 rows and NB blocks of 8 columns at a time
template <int NB, typename Put>
__device__ __noinline__ void product_blocks(int m, int n, int nb, int k, int ks, Mat a, Mat b, Put put) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, g = lane >> 2, t = lane & 3;
  const int steps = (k + 16 * ks - 1) / (16 * ks), wide = (nb + NB - 1) / NB;
  for (int u = warp; u < m / 16 * wide; u += NT / 32) {
    const int i0 = u / wide * 16, j0 = u % wide * 8 * NB;
    float sum[NB][4] = {};
    for (int gg = 0; gg < ks; ++gg) {
      float acc[NB][4] = {};
      for (int st = 0; st < steps; ++st) {
        const int k0 = (gg + st * ks) * 16;
        uint32_t af[4][2], fa[2][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float* p = a.p + (i0 + g + 8 * (i & 1)) * a.rs;
          const int kk = k0 + 2 * (t + 4 * (i >> 1));
          split_pair<2>(kk < k ? p[kk * a.cs] : 0.f, kk + 1 < k ? p[(kk + 1) * a.cs] : 0.f, af[i]);
          fa[0][i] = af[i][0];
          fa[1][i] = af[i][1];
        }
#pragma unroll
        for (int q = 0; q < NB; ++q) {
          uint32_t bf[2][2];
          const int j = j0 + 8 * q + g;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float* p = b.p + j * b.cs;
            const int kk = k0 + 2 * (t + 4 * i);
            const bool ok = j < n;
            split_pair<2>(ok && kk < k ? p[kk * b.rs] : 0.f, ok && kk + 1 < k ? p[(kk + 1) * b.rs] : 0.f,
                          bf[i]);
          }
          mma16816(acc[q], fa[0], bf[0][1], bf[1][1]);
          mma16816(acc[q], fa[1], bf[0][0], bf[1][0]);
          mma16816(acc[q], fa[0], bf[0][0], bf[1][0]);
        }
      }
#pragma unroll
      for (int q = 0; q < NB; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) sum[q][c] = gg ? sum[q][c] + acc[q][c] : acc[q][c];
    }
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int i = i0 + g + 8 * (c >> 1), j = j0 + 8 * q + 2 * t + (c & 1);
        if (j < min(n, 8 * nb)) put(i, j, sum[q][c]);
      }
  }
}

// put(i, j, C(i, j)) for C = A B, A m x k (m a multiple of 16), B k x n; ends with a barrier.
// Where every warp still has work, a fragment of A, loaded and split once, serves two
// blocks of columns (four: no faster, and it spills in the 64 registers that two CTAs on an
// SM leave; one CTA with four blocks is faster up to 152 chains and slower above).
template <typename Put>
__device__ __forceinline__ void product(int m, int n, int k, Mat a, Mat b, Put put) {
  const int ks = groups(m, n, k), steps = (k + 16 * ks - 1) / (16 * ks);
  const bool ext = n == DP;
  const int nb = ext ? D / 8 : (n + 7) / 8, units = m / 16 * nb;
  if (m > 16 && k > 16 && units >= 2 * (NT / 32))
    product_blocks<2>(m, n, nb, k, ks, a, b, put);
  else
    product_blocks<1>(m, n, nb, k, ks, a, b, put);
  if (ext)
    for (int i = threadIdx.x; i < m; i += NT) {
      float sum = 0.f;
      for (int gg = 0; gg < ks; ++gg) {
        float acc = 0.f;
        for (int st = 0; st < steps; ++st)
          for (int kk = (gg + st * ks) * 16; kk < min(k, (gg + st * ks) * 16 + 16); ++kk)
            acc = fmaf(pieces(a.p[i * a.rs + kk * a.cs]), pieces(b.p[kk * b.rs + D * b.cs]), acc);
        sum = gg ? sum + acc : acc;
      }
      put(i, D, sum);
    }
  __syncthreads();
}

__device__ __forceinline__ float warp_sum(float s) {
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

__global__ void __launch_bounds__(NT, 2) k_stack_tail(const __grid_constant__ Args A) {
  __shared__ float xn2[128], rowdot[64], omn[256], den[64], usum[128];
  const int T = A.T, M = A.M, b = A.b, tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const size_t c = blockIdx.x, row0 = c * b;
  float* X = A.scratch + c * A.chain;  // [2][T][64]: q, k
  float* dO = X + 2 * T * D;           // [T][64]
  float* Vx = dO + T * D;              // [T][65]: [V | 1]
  float* W = Vx + T * DP;              // [T][65]
  float* phi = W + T * DP;             // [2][T][M]
  float* dphi = phi + 2 * T * M;       // [2][T][M]
  float* P = dphi + 2 * T * M;         // [M][65]
  float* G = P + M * DP;               // [M][65]
  float* As = G + M * DP;              // [T][T]
  float* dA = As + T * T;              // [T][T]
  float* dV = dA + T * T;              // [T][64]
  float* part = A.part + c * M * D;    // [M][64]
  float *phiQ = phi, *phiK = phi + T * M, *dphiQ = dphi, *dphiK = dphi + T * M;
  if (c == 0 && tid == 0) *A.err = 0;

  for (int e = tid; e < T * D; e += NT) {
    const int r = e / D, j = e % D;
    const size_t s = row0 * D + e;
    const bool ok = r < b;
    X[e] = ok ? __bfloat162float(A.q[s]) : 0.f;
    X[T * D + e] = ok ? __bfloat162float(A.k[s]) : 0.f;
    Vx[r * DP + j] = ok ? __bfloat162float(A.v[s]) : 0.f;
    dO[e] = ok ? __bfloat162float(A.dout[s]) : 0.f;
    if (j == 0) Vx[r * DP + D] = ok ? 1.f : 0.f;
  }
  __syncthreads();
  auto norm2 = [&](const float* x) {
    float s = 0.f;
    for (int j = lane; j < D; j += 32) s = fmaf(x[j], x[j], s);
    return warp_sum(s);
  };
  for (int i = warp; i < 2 * T; i += NT / 32) {
    const float s = norm2(X + i * D);
    if (lane == 0) xn2[i] = s;
  }
  for (int m = warp; m < M; m += NT / 32) {
    const float s = norm2(A.omega + m * D);
    if (lane == 0) omn[m] = sqrtf(s);
  }
  for (int r = warp; r < T; r += NT / 32) {
    float s = 0.f;
    if (r < b)
      for (int j = lane; j < D; j += 32)
        s = fmaf(dO[r * D + j], __bfloat162float(A.out[(row0 + r) * D + j]), s);
    s = warp_sum(s);
    if (lane == 0) rowdot[r] = s;
  }
  __syncthreads();
  {
    // g(Q), g(K): a thread per feature, its Omega row in registers; projections
    // summed in j order, ReLU's sign near zero from a compensated dot product (Dot2)
    const int m = tid % M;
    const float* om = A.omega + m * D;
    float o[D];
#pragma unroll
    for (int j = 0; j < D; ++j) o[j] = om[j];
    const float gamma = 2.f * (float)(D + 2) * 5.9604645e-08f;
    for (int i = tid / M; i < 2 * T; i += NT / M) {
      const float* x = X + i * D;
      float dot = 0.f, f = 0.f;
#pragma unroll
      for (int j = 0; j < D; ++j) dot = fmaf(x[j], o[j], dot);
      if (i % T < b) {
        if (A.feature == SLIM_FEAT_EXP) {
          f = expf(dot - 0.5f * xn2[i]) * A.inv_sqrt_m;
        } else {
          if (fabsf(dot) <= gamma * omn[m] * sqrtf(xn2[i])) {
            float sh = 0.f, sl = 0.f;
            for (int j = 0; j < D; ++j) {
              const float p = __fmul_rn(x[j], om[j]), ep = __fmaf_rn(x[j], om[j], -p);
              float t, e;
              two_sum(sh, p, t, e);
              sh = t;
              sl = __fadd_rn(sl, __fadd_rn(e, ep));
            }
            dot = __fadd_rn(sh, sl);
          }
          f = dot > 0.f ? dot * A.inv_sqrt_m : 0.f;
        }
      }
      phi[i * M + m] = f;
    }
  }
  __syncthreads();

  const Mat mQ{phiQ, M, 1}, mK{phiK, M, 1}, mQt{phiQ, 1, M}, mKt{phiK, 1, M}, mV{Vx, DP, 1}, mW{W, DP, 1};
  // state before the slice (eq. 17)
  product(M, DP, T, mKt, mV, [&](int i, int j, float v) { P[i * DP + j] = v; });
  for (int e = tid; e < M * DP; e += NT) {
    const int m = e / DP, j = e % DP;
    const size_t so = (c * M + m) * D + j, zo = c * M + m;
    float hi = j < D ? A.st.S[so] : A.st.z[zo], lo = 0.f;
    if (j < D ? A.st.S_lo != nullptr : A.st.z_lo != nullptr) lo = j < D ? A.st.S_lo[so] : A.st.z_lo[zo];
    pair_add(hi, lo, -P[e]);
    P[e] = hi + lo;
  }
  __syncthreads();
  product(T, T, M, mQ, Mat{phiK, 1, M}, [&](int i, int j, float v) { As[i * T + j] = j > i ? 0.f : v; });
  product(T, 1, M, mQ, Mat{P + D, DP, 1}, [&](int i, int, float v) { den[i] = v; });
  product(T, 1, T, Mat{As, T, 1}, Mat{Vx + D, DP, 1}, [&](int i, int, float v) { den[i] = v + den[i]; });
  for (int e = tid; e < T * DP; e += NT) {
    const int r = e / DP, j = e % DP;
    float w = 0.f;
    if (r < b && den[r] != 0.f) w = j < D ? dO[r * D + j] / den[r] : -rowdot[r] / den[r];
    W[e] = w;
  }
  __syncthreads();
  product(T, T, DP, mW, Mat{Vx, 1, DP}, [&](int i, int j, float v) { dA[i * T + j] = j > i ? 0.f : v; });
  product(T, M, DP, mW, Mat{P, 1, DP}, [&](int i, int j, float v) { dphiQ[i * M + j] = v; });
  product(T, M, T, Mat{dA, T, 1}, mK, [&](int i, int j, float v) { dphiQ[i * M + j] = v + dphiQ[i * M + j]; });
  // state gradient (eq. 18)
  product(M, DP, T, mQt, mW, [&](int i, int j, float v) { G[i * DP + j] = v; });
  for (int e = tid; e < M * DP; e += NT) {
    const int m = e / DP, j = e % DP;
    const size_t so = (c * M + m) * D + j, zo = c * M + m;
    float hi = 0.f, lo = 0.f;
    if (A.gio.S_in) hi = j < D ? A.gio.S_in[so] : A.gio.z_in[zo];
    const float x = G[e];
    G[e] = hi + lo;
    pair_add(hi, lo, x);
    if (A.gio.S_out) (j < D ? A.gio.S_out[so] : A.gio.z_out[zo]) = hi;
  }
  __syncthreads();
  product(T, M, T, Mat{dA, 1, T}, mQ, [&](int i, int j, float v) { dphiK[i * M + j] = v; });
  product(T, M, DP, mV, Mat{G, 1, DP}, [&](int i, int j, float v) { dphiK[i * M + j] = v + dphiK[i * M + j]; });
  product(T, D, T, Mat{As, 1, T}, mW, [&](int i, int j, float v) { dV[i * D + j] = v; });
  product(T, D, M, mK, Mat{G, DP, 1}, [&](int i, int j, float v) {
    if (i < b) A.dv[(row0 + i) * D + j] = __float2bfloat16_rn(v + dV[i * D + j]);
  });
  // u = dphi (.) g', row sums
  for (int i = warp; i < 2 * T; i += NT / 32) {
    float s = 0.f;
    for (int m = lane; m < M; m += 32) {
      const float f = phi[i * M + m], x = dphi[i * M + m];
      const float u = A.feature == SLIM_FEAT_EXP ? x * f : (f > 0.f ? x * A.inv_sqrt_m : 0.f);
      dphi[i * M + m] = u;
      s += u;
    }
    s = warp_sum(s);
    if (lane == 0) usum[i] = s;
  }
  __syncthreads();
  const Mat mO{const_cast<float*>(A.omega), D, 1};
  const bool ex = A.feature == SLIM_FEAT_EXP;
  for (int side = 0; side < 2; ++side) {
    __nv_bfloat16* dst = (side ? A.dk : A.dq) + row0 * D;
    const float *x = X + side * T * D, *us = usum + side * T;
    product(T, D, M, Mat{dphi + side * T * M, M, 1}, mO, [&](int i, int j, float v) {
      if (ex) v -= x[i * D + j] * us[i];
      if (i < b) dst[i * D + j] = __float2bfloat16_rn(v);
    });
  }
  product(M, D, T, Mat{dphiQ, 1, M}, Mat{X, D, 1}, [&](int i, int j, float v) { part[i * D + j] = v; });
  product(M, D, T, Mat{dphiK, 1, M}, Mat{X + T * D, D, 1},
          [&](int i, int j, float v) { part[i * D + j] = v + part[i * D + j]; });
}

// dOmega: the chains' partials in order, compensated (TwoSum)
__global__ void k_tail_domega(const float* part, float* domega, int chains, int MD) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= MD) return;
  float s = 0.f, c = 0.f;
  for (int i = 0; i < chains; ++i) {
    float t, err;
    two_sum(s, part[(size_t)i * MD + e], t, err);
    s = t;
    c += err;
  }
  domega[e] = s + c;
}

size_t chain_floats(int T, int M) {
  return ((size_t)T * D * 4 + (size_t)T * DP * 2 + (size_t)T * M * 4 + (size_t)M * DP * 2 + (size_t)T * T * 2 + 63) /
         64 * 64;
}
int padded(const Problem& p) { return (p.L + 15) / 16 * 16; }

}  // namespace

bool supports(const Problem& p) {
  return p.dtype == SLIM_BF16 && p.d == D && (p.M == 128 || p.M == 256) &&
         p.feature != SLIM_FEAT_SQUARE && p.L >= 1 && p.L < 64 && p.C >= p.L;
}

size_t workspace_bytes(const Problem& p) {
  Carver cv(nullptr);
  cv.take<int>(64);
  cv.take<float>((size_t)p.chains() * chain_floats(padded(p), p.M));
  cv.take<float>((size_t)p.chains() * p.M * D);
  return cv.bytes();
}

slim_status bwd(const Problem& p, const void* q, const void* k, const void* v, const float* omega,
                const void* out, const void* dout, const StateIn& st, const GradIO& gio, void* dq,
                void* dk, void* dv, float* domega, void* workspace, cudaStream_t s) {
  typedef __nv_bfloat16 bf;
  Carver cv(workspace);
  Args A{};
  A.err = cv.take<int>(64);
  A.b = p.L;
  A.T = padded(p);
  A.M = p.M;
  A.chain = chain_floats(A.T, A.M);
  A.scratch = cv.take<float>((size_t)p.chains() * A.chain);
  A.part = cv.take<float>((size_t)p.chains() * p.M * D);
  A.q = static_cast<const bf*>(q);
  A.k = static_cast<const bf*>(k);
  A.v = static_cast<const bf*>(v);
  A.out = static_cast<const bf*>(out);
  A.dout = static_cast<const bf*>(dout);
  A.omega = omega;
  A.st = st;
  A.gio = gio;
  A.dq = static_cast<bf*>(dq);
  A.dk = static_cast<bf*>(dk);
  A.dv = static_cast<bf*>(dv);
  A.feature = p.feature;
  A.inv_sqrt_m = (float)(1.0 / sqrt((double)p.M));
  {
    prof::Scope ps(prof::K_TILE_BWD_Q, s);
    k_stack_tail<<<p.chains(), NT, 0, s>>>(A);
  }
  if (cudaGetLastError() != cudaSuccess) return SLIM_ERR_CUDA;
  prof::Scope ps(prof::K_REDUCE, s);
  k_tail_domega<<<(p.M * D + 255) / 256, 256, 0, s>>>(A.part, domega, p.chains(), p.M * D);
  return cudaGetLastError() == cudaSuccess ? SLIM_OK : SLIM_ERR_CUDA;
}

}  // namespace tail
}  // namespace slim
