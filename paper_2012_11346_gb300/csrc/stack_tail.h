// Backward of one bf16 slice of fewer than 64 rows in the layer stack; see stack_tail.cu.
#pragma once
#include "common.cuh"

namespace slim {
namespace tail {

// d = 64, M in {128, 256}, exp or ReLU features, fewer than 64 rows in one slice
bool supports(const Problem& p);
size_t workspace_bytes(const Problem& p);
slim_status bwd(const Problem& p, const void* q, const void* k, const void* v, const float* omega,
                const void* out, const void* dout, const StateIn& st, const GradIO& gio, void* dq,
                void* dk, void* dv, float* domega, void* workspace, cudaStream_t s);

}  // namespace tail
}  // namespace slim
