// k_stencil in FP32 (mixed precision), every instance (stencil.cuh)
#define GRMHD_STENCIL_INSTANCE
#include "stencil.cuh"

namespace grmhd {

template cudaError_t stencil_launch<false, float, false>(const Dims&, const PrimIn<float>&, CP3, const double*,
    const double*, const FluxOut<float>*, double* const (*)[3], double* const*, int, cudaStream_t);
template cudaError_t stencil_launch<false, float, true>(const Dims&, const PrimIn<float>&, CP3, const double*,
    const double*, const FluxOut<float>*, double* const (*)[3], double* const*, int, cudaStream_t);
template cudaError_t stencil_launch<true, float, false>(const Dims&, const PrimIn<float>&, CP3, const double*,
    const double*, const FluxOut<float>*, double* const (*)[3], double* const*, int, cudaStream_t);
template cudaError_t stencil_launch<true, float, true>(const Dims&, const PrimIn<float>&, CP3, const double*,
    const double*, const FluxOut<float>*, double* const (*)[3], double* const*, int, cudaStream_t);

GRMHD_OOB_READER(oob_stencil32)

}  // namespace grmhd
