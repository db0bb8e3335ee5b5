// The implicit solve of a stage (Sec. 2.4): k_implicit (staggered q_B) and k_implicit_cc
// (cell-centred q_B, the GLM variant).  The per-cell body is implicit_item (items.cuh).
#include "grmhd_device.cuh"
#include "items.cuh"
#include "kernels.h"
#include "launch.cuh"

namespace grmhd {

// Five blocks per SM (96 registers, about 1 KB of spills): against four (128 registers)
// the mixed-precision and metric instances ran 1.5-4 % faster (512^2 vortex mixed 58.1 ->
// 57.3 us, 128^3 star mixed 398 -> 381 us, FP64 455 -> 442 us per launch); the flat FP64
// instance is unchanged (79.3 us).
template <bool M, bool ACC>
__global__ void __launch_bounds__(128, 5) k_implicit(Dims g, ImpArgs a)
{
    grid_dep_sync();
    const long long tot = (long long)g.n[0] * g.n[1] * g.n[2];
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x)
        implicit_item<M, false, ACC>(g, a, t);
}

// the same solve with cell-centred q_B (GLM variant, Sec. 3.1)
template <bool M>
__global__ void __launch_bounds__(128, 4) k_implicit_cc(Dims g, ImpArgs a)
{
    grid_dep_sync();
    const long long tot = (long long)g.n[0] * g.n[1] * g.n[2];
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x)
        implicit_item<M, true>(g, a, t);
}

cudaError_t launch_implicit(const Dims& g, const ImpArgs& a, int nsm, cudaStream_t st)
{
    const long long work = (long long)g.n[0] * g.n[1] * g.n[2];
    const bool m = a.psi || a.alp;
    if (a.dwacc) launch_k(m ? k_implicit<true, true> : k_implicit<false, true>, grid_for(work, 128, nsm), 128, st, g, a);
    else launch_k(m ? k_implicit<true, false> : k_implicit<false, false>, grid_for(work, 128, nsm), 128, st, g, a);
    return cudaGetLastError();
}

cudaError_t launch_implicit_cc(const Dims& g, const ImpArgs& a, int nsm, cudaStream_t st)
{
    const long long work = (long long)g.n[0] * g.n[1] * g.n[2];
    // GLM contexts are FP64 only: the FP64 residual accepts the root
    launch_k(a.psi || a.alp ? k_implicit_cc<true> : k_implicit_cc<false>, grid_for(work, 128, nsm), 128, st, g,
             a);
    return cudaGetLastError();
}

GRMHD_OOB_READER(oob_implicit)

}  // namespace grmhd
