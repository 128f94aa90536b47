// Single-launch forward of a few rows; see simt_short.cu.
#pragma once
#include "common.cuh"

namespace slim {
namespace simt {

// Rows of a call that k_short takes: one 16-row tile, whose features in pieces just fit beside
// Omega (d = 128, M = 256, fp32: 219,328 of 232,448 bytes).  From 17 rows on the four launches of the
// general sequence serve it: 64 chains, M = 256, bf16, d = 64 19 us for 16 rows, 49 for 17 and 51
// for 48; fp32, d = 128 34, 84 and 82 us.
constexpr int kShortMax = 16;

// The forward of p.L <= kShortMax rows in one slice (C >= L); ks_n, ks_a: the
// reduction groups of a 16-row tile's products (simt_path.cu).  Clears *err.
cudaError_t launch_short(const Problem& p, int ks_n, int ks_a, const void* q, const void* k,
                         const void* v, const float* omega, void* out, const StateOut& st,
                         const StateInit& init, int* err, cudaStream_t s);

}  // namespace simt
}  // namespace slim
