// The fp32-compute path's small kernels: Omega's operand pieces, and the state
// carried over the tiles of a launch sequence.
#include "profiler.h"
#include "simt_tiles.h"
#include "warp_mma.cuh"

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

// One thread per (chain, 4 consecutive state elements): the tiles are loaded
// KB at a time so that their latencies overlap, then folded in order into the
// value/error pair (TwoSum), so that rolling back by subtraction (eq. 17) in
// the reverse order of the additions returns the forward's state to within the
// pair's precision.  Bound by the tile totals' traffic through L2.
namespace {
constexpr int KB = 16;
__device__ __forceinline__ void pair_add4(float4& h, float4& l, const float4& x) {
  pair_add(h.x, l.x, x.x);
  pair_add(h.y, l.y, x.y);
  pair_add(h.z, l.z, x.z);
  pair_add(h.w, l.w, x.w);
}
__device__ __forceinline__ float4 pair_val4(const float4& h, const float4& l) {
  return make_float4(h.x + l.x, h.y + l.y, h.z + l.z, h.w + l.w);
}
__device__ __forceinline__ float4 neg4(const float4& x) { return make_float4(-x.x, -x.y, -x.z, -x.w); }
}  // namespace

__global__ void k_carry(float4* buf, float4* hi_p, float4* lo_p, int chains, int nt, int per, int M,
                        int d, int mode, int first, StateInit init, StateOut out) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int S4 = M * d / 4, E4 = S4 + M / 4;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)chains * E4) return;
  const int c = (int)(idx / E4), e = (int)(idx % E4);
  // this element's place in a caller's (S, z) pair of arrays
  const bool in_s = e < S4;
  const size_t so = in_s ? (size_t)c * S4 + e : (size_t)c * (M / 4) + (e - S4);
  float4 hi = make_float4(0.f, 0.f, 0.f, 0.f), lo = hi;
  if (!first) {
    hi = hi_p[idx];
    lo = lo_p[idx];
  } else if (init.S) {
    hi = reinterpret_cast<const float4*>(in_s ? init.S : init.z)[so];
    const float* il = in_s ? init.S_lo : init.z_lo;
    if (il) lo = reinterpret_cast<const float4*>(il)[so];
  }
  float4* col = buf + (size_t)c * nt * E4 + e;
  if (mode == CARRY_GREV || mode == CARRY_ROLLBACK) {
    for (int t0 = nt - 1; t0 >= 0; t0 -= KB) {
      float4 x[KB];
#pragma unroll
      for (int k = 0; k < KB; ++k)
        if (t0 - k >= 0) x[k] = col[(size_t)(t0 - k) * E4];
#pragma unroll
      for (int k = 0; k < KB; ++k)
        if (t0 - k >= 0) {
          if (mode == CARRY_GREV) col[(size_t)(t0 - k) * E4] = pair_val4(hi, lo);
          pair_add4(hi, lo, mode == CARRY_GREV ? x[k] : neg4(x[k]));
        }
    }
    hi_p[idx] = hi;
    lo_p[idx] = lo;
  }
  if (mode != CARRY_GREV) {
    for (int t0 = 0; t0 < nt; t0 += KB) {
      float4 x[KB];
#pragma unroll
      for (int k = 0; k < KB; ++k)
        if (t0 + k < nt) x[k] = col[(size_t)(t0 + k) * E4];
#pragma unroll
      for (int k = 0; k < KB; ++k)
        if (t0 + k < nt) {
          if (mode == CARRY_FWD || (mode == CARRY_ROLLBACK && (t0 + k) % per == 0))
            col[(size_t)(t0 + k) * E4] = pair_val4(hi, lo);
          pair_add4(hi, lo, x[k]);
        }
    }
  }
  if (mode == CARRY_FWD || mode == CARRY_SUM) {
    hi_p[idx] = hi;
    lo_p[idx] = lo;
  }
  if (out.S) {
    reinterpret_cast<float4*>(in_s ? out.S : out.z)[so] = hi;
    float* ol = in_s ? out.S_lo : out.z_lo;
    if (ol) reinterpret_cast<float4*>(ol)[so] = lo;
  }
}

cudaError_t launch_carry(cudaStream_t s, float* buf, float* hi, float* lo, int chains, int nt,
                         int per, int M, int d, CarryMode mode, bool first, const StateInit& init,
                         const StateOut& out) {
  const long long n = (long long)chains * (M * (d + 1) / 4);
  prof::Scope ps(prof::K_SCAN, s, 0.0, (double)n * 16.0 * (2.0 * nt + 4.0));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((n + 255) / 256));
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_carry, reinterpret_cast<float4*>(buf),
                            reinterpret_cast<float4*>(hi), reinterpret_cast<float4*>(lo), chains, nt,
                            per, M, d, (int)mode, first ? 1 : 0, init, out);
}

// 16 float4 columns per CTA, 16 runs of partials each summed by one thread
// (independent loads in flight: the partials come from L2), the runs then in
// order.
__global__ void __launch_bounds__(256) k_domega(const float4* slots, int n, float* domega, int M, int d) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
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
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(M * d / 64));
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_domega, reinterpret_cast<const float4*>(slots), n, domega, M, d);
}

}  // namespace simt
}  // namespace slim
