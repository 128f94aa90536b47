// Single-launch forward of a few rows; see simt_short.cu.
#pragma once
#include "common.cuh"

namespace slim {
namespace simt {

constexpr int kShortMax = 16;  // rows

// The forward of p.L <= kShortMax rows in one slice (C >= L); ks_n, ks_a: the
// reduction groups of a 16-row tile's products (simt_path.cu).  Clears *err.
cudaError_t launch_short(const Problem& p, int ks_n, int ks_a, const void* q, const void* k,
                         const void* v, const float* omega, void* out, const StateOut& st,
                         const StateInit& init, int* err, cudaStream_t s);

}  // namespace simt
}  // namespace slim
