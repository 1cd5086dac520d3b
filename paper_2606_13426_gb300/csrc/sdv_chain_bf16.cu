// sdv_chain_bf16.cu - the cluster kernels of bfloat16 windows (sdv_chain.cuh).
#include "sdv_chain.cuh"

namespace sdv {

template cudaError_t launch_chain<__nv_bfloat16>(const VerifyArgs&, int, int, int, int, bool, cudaStream_t, bool*);
template cudaError_t launch_finish_long<__nv_bfloat16>(const VerifyArgs&, int, int, bool, cudaStream_t);
template cudaError_t launch_ratios<__nv_bfloat16>(const VerifyArgs&, int, int, int, int, cudaStream_t);

}  // namespace sdv
