// The implicit solve of a stage (Sec. 2.4): k_implicit (staggered q_B) and k_implicit_cc
// (cell-centred q_B, the GLM variant).  The per-cell body is implicit_item (items.cuh).
#include "grmhd_device.cuh"
#include "items.cuh"
#include "kernels.h"
#include "launch.cuh"

namespace grmhd {

// Seven blocks per SM (72 registers, 140-220 B of spills): the solve waits on its loads and
// on dependent arithmetic, so more warps pay until the spills do not.  us per launch at
// five / six / seven / eight blocks: 512^2 vortex FP64 65.7 / 61.7 / 60.3 / 61.2, mixed 44.6 /
// 44.3 / 42.4 / 43.4; 96^3 star mixed 147 / 144 / 148 / 149.  (With the FP64 iteration inlined
// in the kernel and the constants split at every residual it took 79.6 and 57.3 us at five
// blocks, and 168 us; 128^3 star FP64 398 us, 280 now.)  The arguments are grid constants
// because implicit_general takes them by reference: as plain parameters every thread copied
// them to its stack.
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

// The dynamo form (xi != 0): every cell takes the general solve, inline and with the registers
// that its FP64 iteration wants (96, five blocks per SM).  As a call from k_implicit's 72
// registers it was slower: 384^2 FP64 152 against 184 us, mixed 158 / 182, 64^3 with a metric
// 287 / 305, 1-D of 4096 cells 45 / 52.
template <bool M, bool CC, bool ACC>
__global__ void __launch_bounds__(128, CC ? 4 : 5) k_implicit_dynamo(const __grid_constant__ Dims g,
                                                                    const __grid_constant__ ImpArgs a)
{
    grid_dep_sync();
    const long long tot = (long long)g.n[0] * g.n[1] * g.n[2];
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x)
        implicit_solve<M, CC, ACC, true>(g, a, t, false, 0.0, 0.0, 0.0);
}

template <bool M, bool ACC>
static auto implicit_kernel(const ImpArgs& a)
{
    return a.xi != 0.0 ? k_implicit_dynamo<M, false, ACC> : k_implicit<M, ACC>;
}

template <bool M>
static auto implicit_kernel_cc(const ImpArgs& a)
{
    return a.xi != 0.0 ? k_implicit_dynamo<M, true, false> : k_implicit_cc<M>;
}

cudaError_t launch_implicit(const Dims& g, const ImpArgs& a, int nsm, cudaStream_t st)
{
    const long long work = (long long)g.n[0] * g.n[1] * g.n[2];
    const bool m = a.psi || a.alp;
    const int b = grid_for(work, 128, nsm);
    if (a.dwacc) launch_k(m ? implicit_kernel<true, true>(a) : implicit_kernel<false, true>(a), b, 128, st, g, a);
    else launch_k(m ? implicit_kernel<true, false>(a) : implicit_kernel<false, false>(a), b, 128, st, g, a);
    return cudaGetLastError();
}

cudaError_t launch_implicit_cc(const Dims& g, const ImpArgs& a, int nsm, cudaStream_t st)
{
    const long long work = (long long)g.n[0] * g.n[1] * g.n[2];
    // GLM contexts are FP64 only: the FP64 residual accepts the root
    launch_k(a.psi || a.alp ? implicit_kernel_cc<true>(a) : implicit_kernel_cc<false>(a), grid_for(work, 128, nsm), 128,
             st, g, a);
    return cudaGetLastError();
}

GRMHD_OOB_READER(oob_implicit)

}  // namespace grmhd
