// k_stencil in FP64: flat metric, MC (stencil.cuh)
#define GRMHD_STENCIL_INSTANCE
#include "stencil.cuh"

namespace grmhd {

template cudaError_t stencil_launch<false, double, false>(const Dims&, const PrimIn<double>&, CP3, const double*,
    const double*, const FluxOut<double>*, double* const (*)[3], double* const*, int, cudaStream_t);

GRMHD_OOB_READER(oob_stencil64)

}  // namespace grmhd
