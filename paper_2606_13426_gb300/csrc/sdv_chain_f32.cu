// sdv_chain_f32.cu - the cluster kernels of float32 windows (sdv_chain.cuh).
#include "sdv_chain.cuh"

namespace sdv {

template cudaError_t launch_chain<float>(const VerifyArgs&, int, int, int, int, bool, cudaStream_t, bool*);
template cudaError_t launch_finish_long<float>(const VerifyArgs&, int, int, bool, cudaStream_t);
template cudaError_t launch_ratios<float>(const VerifyArgs&, int, int, int, int, cudaStream_t);

}  // namespace sdv
