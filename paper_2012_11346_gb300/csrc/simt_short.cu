// The causal forward of a few rows (L <= 16, one slice) on a running state, in one
// launch: a token or a short segment appended to a stream.
//
// One CTA per chain.  Such a call is bound by latency: as the general sequence of
// four launches it took 70 us for one row of 64 chains (d = 64, M = 256, bf16), where
// its traffic (the state in and out, 8.6 MB) is 1.3 us; in one launch it
// takes 13 us, most of it the host's call.  The arithmetic is that of one 16-row
// tile of the general kernels (simt_tiles.cuh), the same sums in the same order, the bound
// of ReLU's recheck included, so the results are the same bits and a backward may follow.
#include <math.h>

#include "simt_short.h"
#include "tile_math.cuh"

namespace slim {
namespace simt {
namespace {

template <typename IO, int D>
struct ShortSmem {
  static constexpr int NX = Pieces<IO>::NX, NS = Pieces<IO>::NS, OP = D + 4, PV = D + 8, PA = 24;
  static constexpr int threads = 512;
  static constexpr int xs = 2 * 16 * OP, as = NS * 16 * PA, v = NX * 16 * PV;
  // Omega, then the partial sums of the products
  static constexpr int om(int M) { return M * OP > red() ? M * OP : red(); }
  static constexpr int red() { return 4 * 16 * (D + 1) + 8 * 256; }
  static constexpr int bytes(int M) {
    return (om(M) + xs + 2 * 16 + 16 + M) * 4 + (as + v + 2 * NS * 16 * (M + 8)) * 2;
  }
};

struct ShortArgs {
  const void *q, *k, *v;
  const float* omega;
  void* o;
  StateInit init;
  StateOut st;
  int* err;
  int L, M, om_words;  // om_words: floats of the Omega / sums area
  int feature, ks_n, ks_a;
  float inv_sqrt_m;
};

template <typename IO, int D>
__global__ void __launch_bounds__(ShortSmem<IO, D>::threads) k_short(const __grid_constant__ ShortArgs A) {
  using S = ShortSmem<IO, D>;
  constexpr int NX = S::NX, NS = S::NS, OP = S::OP, PV = S::PV, PA = S::PA;
  constexpr bool ZM = D < 64;
  constexpr int NT = S::threads, NW = NT / 32;
  extern __shared__ uint4 smem_raw[];
  const int MP = A.M + 8;
  float* om = reinterpret_cast<float*>(smem_raw);  // [M][OP]
  float* xs = om + A.om_words;                     // [2][16][OP]: q, k
  float* norm2 = xs + S::xs;                       // [2][16]
  float* den_s = norm2 + 32;                       // [16]
  float* zf = den_s + 16;                          // [M]: the state's z (d >= 64: rounded to the pieces)
  bf16* Pq = reinterpret_cast<bf16*>(zf + A.M);    // [NS][16][MP]
  bf16* Pk = Pq + NS * 16 * MP;
  bf16* Vs = Pk + NS * 16 * MP;  // [NX][16][PV]
  bf16* As = Vs + S::v;          // [NS][16][PA]
  float* rn = om;                // [groups][16][D + 1]
  float* ra = rn + 4 * 16 * (D + 1);  // [groups][256]
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, g = lane >> 2, t = lane & 3;
  const int c = blockIdx.x, M = A.M;
  const size_t MD = (size_t)M * D;
  pdl_wait();
  pdl_launch();
  if (c == 0 && tid == 0) *A.err = 0;
  const IO* qg = static_cast<const IO*>(A.q) + (size_t)c * A.L * D;
  const IO* kg = static_cast<const IO*>(A.k) + (size_t)c * A.L * D;
  const IO* vg = static_cast<const IO*>(A.v) + (size_t)c * A.L * D;
  const bool square = A.feature == SLIM_FEAT_SQUARE;
  const float* Si = A.init.S ? A.init.S + c * MD : nullptr;
  const float* Sl = A.init.S_lo ? A.init.S_lo + c * MD : nullptr;
  const float* zi = A.init.S ? A.init.z + (size_t)c * M : nullptr;
  const float* zl = A.init.z_lo ? A.init.z_lo + (size_t)c * M : nullptr;

  // This warp's part of the state, in registers from the start to the end: up to
  // 8 blocks of 16 columns x 16 features.  The block's values are at once the
  // readout's B fragments and, transposed, the layout of the products that update
  // it.  Blocks (columns n16, reduction group gr) of one or two pairs, the group's
  // k16 steps gr, gr + ks_n, ... in turn.
  const int pairs = A.ks_n * (D / 16), two = pairs > NW;
  auto pair_of = [&](int u) { return two ? warp + NW * (u >> 2) : warp; };
  const int sh = A.ks_n == 4 ? 2 : A.ks_n - 1;  // ks_n = 1, 2 or 4
  auto col_of = [&](int u) { return 16 * (pair_of(u) >> sh); };
  auto group_of = [&](int u) { return pair_of(u) & (A.ks_n - 1); };
  auto step_of = [&](int u) { return group_of(u) + ((two ? u & 3 : u) << sh); };
  auto live = [&](int u) { return pair_of(u) < pairs && step_of(u) < M / 16; };
  auto elem = [&](int u, int i) {  // place of element i of block u in S
    const int f = 16 * step_of(u) + 2 * t + (i & 1) + 8 * (i >> 2);
    return (size_t)f * D + col_of(u) + g + 8 * ((i >> 1) & 1);
  };
  float hi[8][8] = {};
  if (Si) {
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (live(u)) {
#pragma unroll
        for (int i = 0; i < 8; ++i) hi[u][i] = Si[elem(u, i)];
      }
  }

  if (!square)
    for (int e = tid; e < M * (D / 4); e += NT) {
      const int m = e / (D / 4), j = e % (D / 4) * 4;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(om + m * OP + j)),
                   "l"(A.omega + (size_t)m * D + j)
                   : "memory");
    }
  cp_commit();
  for (int e = tid; e < 3 * 16 * (D / 8); e += NT) {
    const int w = e / (16 * (D / 8)), r = e / (D / 8) % 16, c8 = e % (D / 8) * 8;
    float v[8] = {};
    if (r < A.L) load8((w == 0 ? qg : w == 1 ? kg : vg) + r * D + c8, v);
    if (w == 2) {
      store_pieces8<NX>(Vs + r * PV + c8, 16 * PV, v);
    } else {
      float4* d = reinterpret_cast<float4*>(xs + (w * 16 + r) * OP + c8);
      d[0] = make_float4(v[0], v[1], v[2], v[3]);
      d[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
  }
  if (zi)
    for (int m = tid; m < M; m += NT) {
      const float z = zi[m] + (zl ? zl[m] : 0.f);
      zf[m] = ZM ? z : round_pieces<NS>(z);
    }
  __syncthreads();
  for (int r = warp; r < 32; r += NW) {
    const float s = warp_norm2<D>(xs + r * OP);
    if (lane == 0) norm2[r] = s;
  }
  cp_wait<0>();
  __syncthreads();

  // g(Q), g(K): an item is one feature of one side, four rows at a time
  for (int it = tid; it < 2 * M; it += NT) {
    const int side = it >= M, m = it - side * M;
    const float* x = xs + side * 16 * OP;
    const float* o = om + m * OP;
    bf16* dst = (side ? Pk : Pq) + m;
    // |omega| in k_setup's order: the bound on a projection's error is then the same number
    // as in the kernels of a backward that follows, and so is every decision
    const float on = A.feature == SLIM_FEAT_RELU ? sqrtf(thread_norm2<D>(o)) : 0.f;
    for (int r0 = 0; r0 < 16; r0 += 4) {
      float acc[4] = {};
      if (r0 < A.L) {
        if (square) {
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[i] = x[(r0 + i) * OP + m] * x[(r0 + i) * OP + m];
        } else {
#pragma unroll 4
          for (int j = 0; j < D; j += 4) {
            const float4 w = *reinterpret_cast<const float4*>(o + j);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 y = *reinterpret_cast<const float4*>(x + (r0 + i) * OP + j);
              acc[i] = fmaf(y.x, w.x, acc[i]);
              acc[i] = fmaf(y.y, w.y, acc[i]);
              acc[i] = fmaf(y.z, w.z, acc[i]);
              acc[i] = fmaf(y.w, w.w, acc[i]);
            }
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
            acc[i] = r0 + i < A.L ? feature_fp<D>(A.feature, acc[i], norm2[side * 16 + r0 + i], on,
                                                  A.inv_sqrt_m, x + (r0 + i) * OP, o, 1)
                                  : 0.f;
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float pc[NS];
        split_bf16<NS>(acc[i], pc);
#pragma unroll
        for (int p = 0; p < NS; ++p) dst[(p * 16 + r0 + i) * MP] = __float2bfloat16_rn(pc[p]);
      }
    }
  }
  __syncthreads();

  // the scores, a reduction group per warp
  for (int u = warp; u < A.ks_a; u += NW) {
    float d0[4] = {}, d1[4] = {};
    for (int s = u; s < M / 16; s += A.ks_a) {
      uint32_t a[NS][4], b[NS][4];
      ld_a<NS>(a, Pq, 16 * MP, MP, 0, 16 * s);
      ld_b<NS>(b, Pk, 16 * MP, MP, 0, 16 * s);
      mma_pieces<NS, NS>(d0, d1, a, b);
    }
    float* dst = ra + u * 256 + 2 * t;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      dst[(g + 8 * h) * 16] = d0[2 * h];
      dst[(g + 8 * h) * 16 + 1] = d0[2 * h + 1];
      dst[(g + 8 * h) * 16 + 8] = d1[2 * h];
      dst[(g + 8 * h) * 16 + 9] = d1[2 * h + 1];
    }
  }
  if (Si) {  // the readout of the state, g(Q) [S | z]
    float d0[4] = {}, d1[4] = {};
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (live(u)) {
        uint32_t a[NS][4], b[NS][4];
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = hi[u][i] + (Sl ? Sl[elem(u, i)] : 0.f);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          uint32_t w0[NS], w1[NS];
          split_pair<NS>(x[2 * q], x[2 * q + 1], w0);
          split_pair<NS>(x[4 + 2 * q], x[5 + 2 * q], w1);
#pragma unroll
          for (int p = 0; p < NS; ++p) {
            b[p][2 * q] = w0[p];
            b[p][2 * q + 1] = w1[p];
          }
        }
        ld_a<NS>(a, Pq, 16 * MP, MP, 0, 16 * step_of(u));
        mma_pieces<NS, NS>(d0, d1, a, b);
        const bool last = u == 7 || (two && u == 3) || !live(u + 1);
        if (last) {
          const int n0 = col_of(u);
          float* dst = rn + group_of(u) * 16 * (D + 1);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float* row = dst + (g + 8 * h) * (D + 1) + n0 + 2 * t;
            row[0] = d0[2 * h];
            row[1] = d0[2 * h + 1];
            row[8] = d1[2 * h];
            row[9] = d1[2 * h + 1];
          }
#pragma unroll
          for (int c4 = 0; c4 < 4; ++c4) d0[c4] = d1[c4] = 0.f;
        }
      }
    if (ZM) {  // z as an MMA column, a group per warp
      for (int gr = warp; gr < A.ks_n; gr += NW) {
        float dz[4] = {};
        for (int s = gr; s < M / 16; s += A.ks_n) {
          uint32_t a[NS][4], w0[NS] = {}, w1[NS] = {};
          ld_a<NS>(a, Pq, 16 * MP, MP, 0, 16 * s);
          if (g == 0) {
            const float* z = zf + 16 * s + 2 * t;
            split_pair<NS>(z[0], z[1], w0);
            split_pair<NS>(z[8], z[9], w1);
          }
#pragma unroll
          for (int o = NS - 1; o >= 0; --o)
#pragma unroll
            for (int x = 0; x <= o; ++x) mma16816(dz, a[x], w0[o - x], w1[o - x]);
        }
        if (t == 0) {
          rn[(gr * 16 + g) * (D + 1) + D] = dz[0];
          rn[(gr * 16 + g + 8) * (D + 1) + D] = dz[2];
        }
      }
    } else if (NT - 1 - tid < 16 * A.ks_n) {  // den, feature after feature in each group
      const int r = (NT - 1 - tid) % 16, gr = (NT - 1 - tid) / 16;
      float e = 0.f;
      if (r < A.L)
        for (int s = gr; s < M / 16; s += A.ks_n)
#pragma unroll
          for (int k = 0; k < 16; k += 8) {
            float x[8];
            add_pieces8<NS>(Pq + r * MP + 16 * s + k, 16 * MP, x);
#pragma unroll
            for (int i = 0; i < 8; ++i) e = fmaf(x[i], zf[16 * s + k + i], e);
          }
      rn[(gr * 16 + r) * (D + 1) + D] = e;
    }
  }
  __syncthreads();
  {  // scores: groups in order, mask, pieces
    const int row = tid / 16, key = tid % 16;
    if (tid < 256) {
      float v = ra[tid];
      for (int q = 1; q < A.ks_a; ++q) v += ra[q * 256 + tid];
      float pc[NS];
      split_bf16<NS>(key <= row ? v : 0.f, pc);
#pragma unroll
      for (int p = 0; p < NS; ++p) As[(p * 16 + row) * PA + key] = __float2bfloat16_rn(pc[p]);
    }
  }
  auto grouped = [&](int row, int col) {
    const float* p = rn + row * (D + 1) + col;
    float v = 0.f;
    if (Si) {
      v = p[0];
      for (int q = 1; q < A.ks_n; ++q) v += p[q * 16 * (D + 1)];
    }
    return v;
  };
  __syncthreads();
  if (ZM) {
    if (warp == 0) {
      uint32_t a[NS][4];
      ld_a<NS>(a, As, 16 * PA, PA, 0, 0);
      float d0[4] = {};
      const uint32_t one = g == 0 ? kOnes : 0u;
      mma_n8<NS>(d0, a, one, one);
      if (t == 0) {
        den_s[g] = d0[0] + grouped(g, D);
        den_s[g + 8] = d0[2] + grouped(g + 8, D);
      }
    }
  } else if (tid < 16) {
    float e = 0.f;
    for (int k = 0; k <= tid; ++k) e += staged_sum<NS>(As + tid * PA + k, 16 * PA);
    den_s[tid] = e + grouped(tid, D);
  }
  __syncthreads();
  IO* og = static_cast<IO*>(A.o) + (size_t)c * A.L * D;
  for (int n0 = 16 * warp; n0 < D; n0 += 16 * (NW)) {
    uint32_t a[NS][4], b[NX][4];
    float d[2][4] = {};
    ld_a<NS>(a, As, 16 * PA, PA, 0, 0);
    ld_bt<NX>(b, Vs, 16 * PV, PV, n0, 0);
    mma_pieces<NS, NX>(d[0], d[1], a, b);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = g + 8 * h, col = n0 + 8 * q + 2 * t;
        const float den = den_s[row];
        if (row < A.L) {
          const float x = d[q][2 * h] + grouped(row, col), y = d[q][2 * h + 1] + grouped(row, col + 1);
          store2(og + row * D + col, den != 0.f ? x / den : 0.f, den != 0.f ? y / den : 0.f);
        }
      }
  }

  // the state after the rows (it may be written where it was read: other warps'
  // reads are behind the barriers above)
  auto put = [&](float* hi_o, float* lo_o, float h, float l, size_t e, float v) {
    pair_add(h, l, v);
    hi_o[e] = h;
    if (lo_o) lo_o[e] = l;
  };
  float* So = A.st.S + c * MD;
  float* Lo = A.st.S_lo ? A.st.S_lo + c * MD : nullptr;
  float* zo = A.st.z + (size_t)c * M;
  float* zlo = A.st.z_lo ? A.st.z_lo + (size_t)c * M : nullptr;
#pragma unroll
  for (int u = 0; u < 8; ++u)
    if (live(u)) {  // Delta^T = V^T g(K), the pieces' products in Delta's order
      uint32_t a[NX][4], b[NS][4];
      float d[2][4] = {};
      ld_at<NX>(a, Vs, 16 * PV, PV, col_of(u), 0);
      ld_bt<NS>(b, Pk, 16 * MP, MP, 16 * step_of(u), 0);
#pragma unroll
      for (int o = NS - 1; o >= 0; --o)
#pragma unroll
        for (int i = 0; i <= o; ++i)
          if (o - i < NX) {
            mma16816(d[0], a[o - i], b[i][0], b[i][1]);
            mma16816(d[1], a[o - i], b[i][2], b[i][3]);
          }
      float lo[8] = {};
      if (Sl) {
#pragma unroll
        for (int i = 0; i < 8; ++i) lo[i] = Sl[elem(u, i)];
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) put(So, Lo, hi[u][i], lo[i], elem(u, i), d[i >> 2][i & 3]);
    }
  if (ZM) {
    for (int mb = warp; mb < M / 16; mb += NW) {
      uint32_t a[NS][4];
      ld_at<NS>(a, Pk, 16 * MP, MP, 16 * mb, 0);
      float d[4] = {};
      const uint32_t one = g == 0 ? kOnes : 0u;
      mma_n8<NS>(d, a, one, one);
      if (t == 0) {
        const int f0 = 16 * mb + g;
        put(zo, zlo, zi ? zi[f0] : 0.f, zl ? zl[f0] : 0.f, f0, d[0]);
        put(zo, zlo, zi ? zi[f0 + 8] : 0.f, zl ? zl[f0 + 8] : 0.f, f0 + 8, d[2]);
      }
    }
  } else {
    for (int m = tid; m < M; m += NT) {
      float e = 0.f;
      for (int r = 0; r < A.L; ++r) e += staged_sum<NS>(Pk + r * MP + m, 16 * MP);
      put(zo, zlo, zi ? zi[m] : 0.f, zl ? zl[m] : 0.f, m, e);
    }
  }
}

template <typename IO, int D>
cudaError_t run(const Problem& p, ShortArgs& A, cudaStream_t s) {
  using S = ShortSmem<IO, D>;
  static_assert(S::bytes(256) <= kSmemMax, "shared memory");
  static bool flags[kMaxDevices] = {};
  bool* set = device_flag(flags);
  if (set == nullptr) return cudaErrorInvalidDevice;
  if (!*set) {
    const cudaError_t e = cudaFuncSetAttribute(k_short<IO, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               S::bytes(256));
    if (e != cudaSuccess) return e;
    *set = true;
  }
  A.om_words = S::om(p.M);
  const double rows = (double)p.chains() * p.L;
  prof::Scope ps(prof::K_TILE_OUT, s, (p.feature == SLIM_FEAT_SQUARE ? 4.0 : 8.0) * rows * D * p.M,
                 4.0 * rows * D * sizeof(IO) + 8.0 * p.chains() * p.M * (D + 1));
  return launch_pdl(k_short<IO, D>, (unsigned)p.chains(), S::threads, S::bytes(p.M), s, A);
}

}  // namespace

cudaError_t launch_short(const Problem& p, int ks_n, int ks_a, const void* q, const void* k,
                         const void* v, const float* omega, void* out, const StateOut& st,
                         const StateInit& init, int* err, cudaStream_t s) {
  ShortArgs A{};
  A.q = q;
  A.k = k;
  A.v = v;
  A.omega = omega;
  A.o = out;
  A.init = init;
  A.st = st;
  A.err = err;
  A.L = p.L;
  A.M = p.M;
  A.feature = (int)p.feature;
  A.ks_n = ks_n;
  A.ks_a = ks_a;
  A.inv_sqrt_m = (float)(1.0 / sqrt((double)p.M));
  const bool f = p.dtype == SLIM_F32;
  if (p.d == 16) return f ? run<float, 16>(p, A, s) : run<bf16, 16>(p, A, s);
  if (p.d == 32) return f ? run<float, 32>(p, A, s) : run<bf16, 32>(p, A, s);
  if (p.d == 64) return f ? run<float, 64>(p, A, s) : run<bf16, 64>(p, A, s);
  return f ? run<float, 128>(p, A, s) : run<bf16, 128>(p, A, s);
}

}  // namespace simt
}  // namespace slim
