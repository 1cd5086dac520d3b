// sdv_rounds_c16.cu - the round kernels for mixtures of up to 16 components (sdv_rounds.cuh).
#include "sdv_rounds.cuh"

namespace sdv {

template int launch_rounds_c<16>(const RoundsArgs&, bool, cudaStream_t);

}  // namespace sdv
