// k_stencil in FP64: metric, MC (stencil.cuh)
#define GRMHD_STENCIL_INSTANCE
#include "stencil.cuh"

namespace grmhd {

template cudaError_t stencil_launch<true, double, false>(const Dims&, const PrimIn<double>&, CP3, const double*,
    const double*, const FluxOut<double>*, double* const (*)[3], double* const*, int, cudaStream_t);

GRMHD_OOB_READER(oob_stencil64m)

}  // namespace grmhd
