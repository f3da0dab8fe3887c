// x1 turn (inverse x1 transform, update, forward x1 transform) in float (instantiations).
#include "fftls_turn.cuh"

namespace fftls {

template cudaError_t launch_turn<float>(const IterArgs<float>&, cudaStream_t);
template cudaError_t set_attrs_turn<float>(size_t);
template size_t turn_smem_reg<float>(int, int, int);

}  // namespace fftls
