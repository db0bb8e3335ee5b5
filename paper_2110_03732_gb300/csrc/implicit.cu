// The implicit solve of a stage (Sec. 2.4): k_implicit (staggered q_B) and k_implicit_cc
// (cell-centred q_B, the GLM variant).  The per-cell body is implicit_item (items.cuh).
#include "grmhd_device.cuh"
#include "items.cuh"
#include "kernels.h"
#include "launch.cuh"

namespace grmhd {

// Seven blocks per SM (72 registers, 130-200 B of spills): the solve waits on its loads and
// on dependent arithmetic, so more warps pay until the spills do not.  us per launch at
// five / six / seven / eight blocks: 512^2 vortex FP64 65.7 / 61.7 / 60.3 / 61.2, mixed 44.6 /
// 44.3 / 42.4 / 43.4; 96^3 star mixed 147 / 144 / 148 / 149.  (With the FP64 iteration inlined
// in the kernel and the constants split at every residual it took 79.6 and 57.3 us at five
// blocks, and 168 us; 128^3 star FP64 398 us, 277 now.)  The arguments are grid constants because implicit_general takes
// them by reference: as plain parameters every thread copied them to its stack.
template <bool M, bool ACC>
__global__ void __launch_bounds__(128, 7) k_implicit(const __grid_constant__ Dims g, const __grid_constant__ ImpArgs a)
{
    grid_dep_sync();
    const long long tot = (long long)g.n[0] * g.n[1] * g.n[2];
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x)
        implicit_item<M, false, ACC>(g, a, t);
}

// the same solve with cell-centred q_B (GLM variant, Sec. 3.1); eight blocks: 384^2 vortex
// 40.8 / 39.8 / 39.1 / 37.1 us at five to eight
template <bool M>
__global__ void __launch_bounds__(128, 8) k_implicit_cc(const __grid_constant__ Dims g, const __grid_constant__ ImpArgs a)
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
