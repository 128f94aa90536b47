// Tile kernels of the fp32-compute path (simt_tiles.cuh): launch interface.
#pragma once
#include "common.cuh"

namespace slim {
namespace simt {

constexpr int kTile = 64;  // rows of a frame, and of the largest tile
constexpr int kSms = 152;  // streaming multiprocessors of a GB300

// One launch sequence: rows [a, a + b) of every chain, cut into nt tiles of up to
// `pitch` rows per chain; a frame is `per` consecutive tiles, frame i = chain * nf + i.  A
// state (S, z) is E = M d + M floats, S row-major [M][d], then z.
struct TileArgs {
  const void *q, *k, *v, *out, *dout;  // caller tensors [chains][L][d]
  void *o, *dq, *dk, *dv;
  const float* omega;          // caller's Omega [M][d] fp32 (null for the quadratic map)
  const float* om_t;           // transposed in blocks of 64 features: [M / 64][d][64], zero past M
  const __nv_bfloat16* om_row; // its pieces [3][M][d]
  const float* om_norm;        // |omega_m|
  float* delta;                // [frames][E]: a tile's sum of T_l; with several tiles per frame
                               // [frames][2][E], the frame's sum as a value/error pair
  float* zdelta;               // [tiles][M]: the z part of every tile (several tiles per frame)
  const float* P;              // state of frame i at P + chain * p_chain + i * p_frame; its errors
  long long p_chain, p_frame, p_lo;  // p_lo further (the forward, several tiles per frame)
  float* gdelta;               // [frames][E]: a frame's share of the state gradient
  const float* G;              // state gradient of frame i, as for P
  long long g_chain, g_frame;
  __nv_bfloat16* phi_k;        // [frames][pieces][64][M]: g(K)
  // what the query side of the backward leaves for the key side, in pieces
  __nv_bfloat16 *phi_q;        // [frames][pieces][64][M]: g(Q)
  __nv_bfloat16 *sA, *sdA;     // [frames][pieces][64][64]: scores and their gradient
  __nv_bfloat16 *sW;           // [frames][pieces][64][d]: dout / den
  float* slots;                // dOmega partials, one per CTA
  int slots_new;               // bwd_k starts its partials (bwd_q always does) instead of adding
  int L, M, E, a, b, chains;
  int rows, pitch, per;        // a tile's rows in a frame (16, 32, 48 or 64) and in the sequence; tiles per frame
  int shift;                   // frame row >> shift: the tile of the frame
  int slice, slice_tiles;      // rows and tiles of a slice (tiles start anew in every slice)
  int nt, nf;                  // tiles and frames per chain
  int ks_n, ks_a;              // reduction groups of the readout's and the scores' k16 steps (rows < 48)
  int feature, causal;
  float inv_sqrt_m;
};

// Kernels of one (dtype, d).
struct TileKernels {
  cudaError_t (*delta)(const TileArgs&, cudaStream_t);  // g(K), Delta_t = g(K)^T [V | 1]
  cudaError_t (*out)(const TileArgs&, cudaStream_t);    // g(Q), scores, readout
  cudaError_t (*bwd_q)(const TileArgs&, cudaStream_t);  // query side of the backward
  cudaError_t (*bwd_k)(const TileArgs&, cudaStream_t);  // key / value side
  int slots;  // most CTAs, and dOmega partials, of a backward launch
};
const TileKernels& tile_kernels(slim_dtype dtype, int d);

// Omega's operand forms and norms (skipped when omega is null), the error word
// cleared, dOmega zeroed (when given).
cudaError_t launch_setup(cudaStream_t s, const float* omega, int M, int d, float* om_t,
                         __nv_bfloat16* om_row, float* om_norm, float* domega, int* err);

enum CarryMode {
  CARRY_FWD = 0,       // P_i = B + sum_{i'<i} D_i' (in place), then B += sum_i D_i
  CARRY_SUM = 1,       // B += sum_i D_i only
  CARRY_ROLLBACK = 2,  // B -= sum_i D_i (eq. 17), then P_i as CARRY_FWD, B left rolled back
  CARRY_GREV = 3       // G_i = G + sum_{i'>i} D_i' (in place), then G += sum_i D_i
};
struct CarryArgs {
  float* buf;           // frame totals [chains][nf][E], or pairs [chains][nf][2][E]
  int pairs;
  float *hi, *lo;       // the carried state, a value/error pair [chains][E]
  int chains, nf, M, d;
  CarryMode mode;
  int first;            // the pair starts from `init` (zero when init.S is null) instead of hi / lo
  StateInit init;
  StateOut out;         // out.S non-null: the pair is also written there
};
cudaError_t launch_carry(cudaStream_t s, const CarryArgs& a);

// dOmega += the `n` partials, in a fixed order, compensated (TwoSum).
cudaError_t launch_domega(cudaStream_t s, const float* slots, int n, float* domega, int M, int d);

}  // namespace simt
}  // namespace slim
