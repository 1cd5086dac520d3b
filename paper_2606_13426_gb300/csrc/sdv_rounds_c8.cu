// sdv_rounds_c8.cu - the round kernels for mixtures of up to 8 components (sdv_rounds.cuh).
#include "sdv_rounds.cuh"

namespace sdv {

template int launch_rounds_c<8>(const RoundsArgs&, bool, cudaStream_t);

}  // namespace sdv
