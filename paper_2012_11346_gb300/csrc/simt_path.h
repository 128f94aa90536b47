// fp32-compute path of libslim (fp32 operands, warp-MMA contractions); see simt_path.cu.
#pragma once
#include "common.cuh"

namespace slim {
namespace simt {

// small: the least workspace the forward runs in (fwd takes any size from there
// on, and sweeps fewer rows and chains at a time below the full size)
size_t workspace_bytes(const Problem& p, bool bwd, bool small = false);

// What slim_fwd_noalloc's limit counts: a call's state and the rows of one slice
// (of 1024 rows of shorter slices) with their features and tile totals in fp32.
// This is the size of the problem, not of the scratch: the limit stays where it is
// when the layout of the scratch changes.  fwd runs in less for every problem
// within SLIM_NOALLOC_SCRATCH_BYTES.
size_t noalloc_bytes(const Problem& p);

// out null: the state alone
slim_status fwd(const Problem& p, const void* q, const void* k, const void* v,
                const float* omega, void* out, const StateOut& st, const StateInit& init,
                void* workspace, size_t bytes, cudaStream_t s);

slim_status bwd(const Problem& p, const void* q, const void* k, const void* v,
                const float* omega, const void* out, const void* dout, const StateIn& st,
                const GradIO& gio, void* dq, void* dk, void* dv, float* domega, void* workspace,
                cudaStream_t s);

// The non-causal form (no mask, one global state; S_state/z_state are that
// state), on the same workspace layout as the causal sweeps.
slim_status fwd_bidir(const Problem& p, const void* q, const void* k, const void* v,
                      const float* omega, void* out, const StateOut& st, void* workspace,
                      cudaStream_t s);
slim_status bwd_bidir(const Problem& p, const void* q, const void* k, const void* v,
                      const float* omega, const void* out, const void* dout, const StateIn& st,
                      void* dq, void* dk, void* dv, float* domega, void* workspace,
                      cudaStream_t s);

}  // namespace simt
}  // namespace slim
