// sdv_chain.h - host entries of the cluster kernels (sdv_chain.cuh), for T = float and
// __nv_bfloat16 windows.
#pragma once

#include <cuda_runtime.h>

#include "sdv_host.h"

namespace sdv {

// Launches k_chain when the call fits it (chain_cluster); *taken says whether it did.
template <typename T>
cudaError_t launch_chain(const VerifyArgs& A, int B, int L, int vpt, int rows, bool vec4, cudaStream_t s, bool* taken);

// Launches k_finish_long, the end of a call streamed by k_tiles, for rows too long for
// k_finish, to overlap its predecessor.
template <typename T>
cudaError_t launch_finish_long(const VerifyArgs& A, int B, int L, bool vec4, cudaStream_t s);

// Launches k_ratios, the log ratios alone.
template <typename T>
cudaError_t launch_ratios(const VerifyArgs& A, int B, int L, int vpt, int rows, cudaStream_t s);

}  // namespace sdv
