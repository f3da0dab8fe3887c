// x1 turn (inverse x1 transform, update, forward x1 transform) in double (instantiations).
#include "fftls_turn.cuh"

namespace fftls {

template cudaError_t launch_turn<double>(const IterArgs<double>&, cudaStream_t);
template cudaError_t set_attrs_turn<double>(size_t);
template size_t turn_smem_reg<double>(int, int, int);

}  // namespace fftls
