// The fp32-compute path's small kernels: Omega's operand pieces, and the state
// carried over the tiles of a launch sequence.
#include "simt_tiles.h"
#include "tile_math.cuh"

namespace slim {
namespace simt {

extern const TileKernels kTilesD16F32, kTilesD16Bf16, kTilesD32F32, kTilesD32Bf16, kTilesD64F32,
    kTilesD64Bf16, kTilesD128F32, kTilesD128Bf16;

const TileKernels& tile_kernels(slim_dtype dtype, int d) {
  const bool f = dtype == SLIM_F32;
  if (d == 16) return f ? kTilesD16F32 : kTilesD16Bf16;
  if (d == 32) return f ? kTilesD32F32 : kTilesD32Bf16;
  if (d == 64) return f ? kTilesD64F32 : kTilesD64Bf16;
  return f ? kTilesD128F32 : kTilesD128Bf16;
}

// Omega as the kernels read it: fp32, transposed in blocks of 64 features, for
// the FMA projections; three bf16 pieces (24 bits) for the MMAs; the row norms.
__global__ void k_setup(const float* __restrict__ omega, int M, int d, float* om_t, bf16* om_row,
                        float* om_norm, float* domega, int* err) {
  const int gid = blockIdx.x * blockDim.x + threadIdx.x, gn = gridDim.x * blockDim.x;
  if (gid == 0) *err = 0;
  if (domega)
    for (int e = gid; e < M * d; e += gn) domega[e] = 0.f;
  if (!omega) return;
  for (int e = gid; e < (M + 63) / 64 * 64 * d; e += gn) {
    const int mm = e % 64, j = e / 64 % d, m = e / 64 / d * 64 + mm;
    om_t[e] = m < M ? omega[(size_t)m * d + j] : 0.f;
  }
  for (int e = gid; e < M * d; e += gn) {
    float pc[3];
    split_bf16<3>(omega[e], pc);
#pragma unroll
    for (int p = 0; p < 3; ++p) om_row[(size_t)p * M * d + e] = __float2bfloat16_rn(pc[p]);
  }
  const int lane = threadIdx.x % 32;
  for (int m = gid / 32; m < M; m += gn / 32) {
    float s = 0.f;
    for (int j = lane; j < d; j += 32) s = fmaf(omega[(size_t)m * d + j], omega[(size_t)m * d + j], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) om_norm[m] = sqrtf(s);
  }
}

cudaError_t launch_setup(cudaStream_t s, const float* omega, int M, int d, float* om_t, bf16* om_row,
                         float* om_norm, float* domega, int* err) {
  prof::Scope ps(prof::K_PREP, s);
  k_setup<<<omega || domega ? 64 : 1, 256, 0, s>>>(omega, M, d, om_t, om_row, om_norm, domega, err);
  return cudaGetLastError();
}

// One thread per (chain, V consecutive state elements): the totals are loaded KB at
// a time so that their latencies overlap, then folded in order into the value/error
// pair (TwoSum), so that rolling back by subtraction (eq. 17) in the reverse
// order of the additions returns the forward's state to within the pair's
// precision.  Bound by the totals' traffic, and with few chains by the loads in
// flight: one element per thread there (V = 1), four where the threads fill the chip.
// The totals come one per frame (PAIR false) or as pairs.
namespace {
template <int V> struct Vec;
template <> struct Vec<1> { typedef float T; };
template <> struct Vec<4> { typedef float4 T; };

__device__ __forceinline__ void pair_add2(float& hi, float& lo, float xh, float xl) {
  float s, e;
  two_sum(hi, xh, s, e);
  two_sum(s, __fadd_rn(__fadd_rn(lo, xl), e), hi, lo);
}
}  // namespace

template <int V, int KB, bool PAIR>
__global__ void __launch_bounds__(256) k_carry(const __grid_constant__ CarryArgs A) {
  typedef typename Vec<V>::T T;
  union Reg {
    T v;
    float f[V];
  };
  const int SV = A.M * A.d / V, EV = SV + A.M / V, mode = A.mode;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)A.chains * EV) return;
  const int c = (int)(idx / EV), e = (int)(idx % EV);
  // this element's place in a caller's (S, z) pair of arrays
  const bool in_s = e < SV;
  const size_t so = in_s ? (size_t)c * SV + e : (size_t)c * (A.M / V) + (e - SV);
  T* hi_p = reinterpret_cast<T*>(A.hi);
  T* lo_p = reinterpret_cast<T*>(A.lo);
  Reg hi{}, lo{};
  if (!A.first) {
    hi.v = __ldcg(hi_p + idx);
    lo.v = __ldcg(lo_p + idx);
  } else if (A.init.S) {
    hi.v = reinterpret_cast<const T*>(in_s ? A.init.S : A.init.z)[so];
    const float* il = in_s ? A.init.S_lo : A.init.z_lo;
    if (il) lo.v = reinterpret_cast<const T*>(il)[so];
  }
  pdl_wait();  // the totals; the carried state is older
  pdl_launch();
  const bool rev = mode == CARRY_GREV || mode == CARRY_ROLLBACK;
  // frame i's place in buf
  const size_t fs = (size_t)(PAIR ? 2 : 1) * EV;
  T* col = reinterpret_cast<T*>(A.buf) + (size_t)c * A.nf * fs + e;
  const int n = A.nf;
  // passes over the totals: backwards for G and the rollback, forwards for P
  for (int pass = rev ? 0 : 1; pass < (mode == CARRY_GREV ? 1 : 2); ++pass) {
    const bool neg = pass == 0 && mode == CARRY_ROLLBACK;
    for (int i0 = 0; i0 < n; i0 += KB) {
      Reg x[KB], y[PAIR ? KB : 1];
#pragma unroll
      for (int k = 0; k < KB; ++k)
        if (i0 + k < n) {
          const int i = pass == 0 ? n - 1 - i0 - k : i0 + k;
          x[k].v = col[(size_t)i * fs];
          if (PAIR) y[k].v = col[(size_t)i * fs + EV];
        }
#pragma unroll
      for (int k = 0; k < KB; ++k)
        if (i0 + k < n) {
          const int i = pass == 0 ? n - 1 - i0 - k : i0 + k;
          if (mode != CARRY_SUM && (pass == 1 || mode == CARRY_GREV)) {
            T* dst = col + (size_t)i * fs;
            if (PAIR && mode == CARRY_FWD) {  // the frame's kernel moves on from the pair
              dst[0] = hi.v;
              dst[EV] = lo.v;
            } else {
              Reg p;
#pragma unroll
              for (int j = 0; j < V; ++j) p.f[j] = hi.f[j] + lo.f[j];
              dst[0] = p.v;
            }
          }
#pragma unroll
          for (int j = 0; j < V; ++j) {
            const float xh = neg ? -x[k].f[j] : x[k].f[j];
            if (PAIR)
              pair_add2(hi.f[j], lo.f[j], xh, neg ? -y[k].f[j] : y[k].f[j]);
            else
              pair_add(hi.f[j], lo.f[j], xh);
          }
        }
    }
    // the state to carry on: after the sums, or rolled back (a forward's last state goes to
    // the caller alone)
    if (pass == 0 || (mode != CARRY_ROLLBACK && !(mode == CARRY_FWD && A.out.S))) {
      hi_p[idx] = hi.v;
      lo_p[idx] = lo.v;
    }
  }
  if (A.out.S) {
    reinterpret_cast<T*>(in_s ? A.out.S : A.out.z)[so] = hi.v;
    float* ol = in_s ? A.out.S_lo : A.out.z_lo;
    if (ol) reinterpret_cast<T*>(ol)[so] = lo.v;
  }
}

cudaError_t launch_carry(cudaStream_t s, const CarryArgs& a) {
  const long long n = (long long)a.chains * a.M * (a.d + 1);
  prof::Scope ps(prof::K_SCAN, s, 0.0, (double)n * 4.0 * (2.0 * a.nf + 4.0));
  const bool few = n / 4 < kSms * 64;  // too few threads for the chip with four elements each
  const unsigned grid = (unsigned)((few ? n + 255 : n / 4 + 255) / 256);
  if (a.pairs)
    return few ? launch_pdl(k_carry<1, 16, true>, grid, 256, 0, s, a)
               : launch_pdl(k_carry<4, 8, true>, grid, 256, 0, s, a);
  return few ? launch_pdl(k_carry<1, 16, false>, grid, 256, 0, s, a)
             : launch_pdl(k_carry<4, 8, false>, grid, 256, 0, s, a);
}

// 16 float4 columns per CTA, 16 runs of partials each summed by one thread
// (independent loads in flight: the partials come from L2), the runs then in
// order.
__global__ void __launch_bounds__(256) k_domega(const float4* slots, int n, float* domega, int M, int d) {
  pdl_wait();
  pdl_launch();
  __shared__ float4 sh[2][16][16];
  const int col = threadIdx.x % 16, run = threadIdx.x / 16, n4 = M * d / 4;
  const int e = blockIdx.x * 16 + col;  // M d / 4 is a multiple of 64
  const int per = (n + 15) / 16, i0 = run * per, i1 = min(n, i0 + per);
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f), c = s;
  auto add = [](float& s, float& c, float x) {
    float t, err;
    two_sum(s, x, t, err);
    s = t;
    c += err;
  };
#pragma unroll 8
  for (int i = i0; i < i1; ++i) {
    const float4 x = slots[(size_t)i * n4 + e];
    add(s.x, c.x, x.x);
    add(s.y, c.y, x.y);
    add(s.z, c.z, x.z);
    add(s.w, c.w, x.w);
  }
  sh[0][run][col] = s;
  sh[1][run][col] = c;
  __syncthreads();
  if (threadIdx.x >= 64) return;
  // thread: component k of column cc; the column's 16 x 16 block and lane give (m, j)
  const int cc = threadIdx.x / 4, k = threadIdx.x % 4, el = blockIdx.x * 16 + cc;
  const int lane = el % 32, n8 = (el / 32) % 2, n16 = (el / 64) % (d / 16), mb = el / 64 / (d / 16);
  const int m = 16 * mb + (lane >> 2) + 8 * (k >> 1), j = 16 * n16 + 8 * n8 + 2 * (lane & 3) + (k & 1);
  float S = domega[(size_t)m * d + j], C = 0.f;
  for (int r = 0; r < 16; ++r) {
    add(S, C, reinterpret_cast<const float*>(&sh[0][r][cc])[k]);
    C += reinterpret_cast<const float*>(&sh[1][r][cc])[k];
  }
  domega[(size_t)m * d + j] = S + C;
}

cudaError_t launch_domega(cudaStream_t s, const float* slots, int n, float* domega, int M, int d) {
  prof::Scope ps(prof::K_REDUCE, s, 0.0, (double)n * M * d * 4.0);
  return launch_pdl(k_domega, (unsigned)(M * d / 64), 256, 0, s, reinterpret_cast<const float4*>(slots), n,
                    domega, M, d);
}

}  // namespace simt
}  // namespace slim
