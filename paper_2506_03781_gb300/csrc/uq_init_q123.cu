// The initialization (uq_init.cuh) for q = 1, 2, 3.
#include "uq_init.cuh"

namespace uq {

template cudaError_t launch_init_q<1>(const Shape&, const void*, int, int, int, uq_params, uint8_t*, cudaStream_t);
template cudaError_t launch_init_q<2>(const Shape&, const void*, int, int, int, uq_params, uint8_t*, cudaStream_t);
template cudaError_t launch_init_q<3>(const Shape&, const void*, int, int, int, uq_params, uint8_t*, cudaStream_t);

}  // namespace uq
