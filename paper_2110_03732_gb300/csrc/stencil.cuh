// The explicit stencil of a stage in one launch, k_stencil, and its launcher.  Each
// FP64 instance is a translation unit of its own (stencil64*.cu, the FP32 ones
// stencil32.cu), so that they compile in parallel; a unit that defines
// GRMHD_STENCIL_INSTANCE gets the kernel and the launcher, others the declaration.
#pragma once

#include <cstring>

#include "grmhd_device.cuh"
#include "items.cuh"
#include "kernels.h"
#include "launch.cuh"

namespace grmhd {

// ---------------------------------------------------------------------------
// the explicit stencil of a stage: face fluxes and upwind constrained transport
// (hat{E}_C on the edges along C, stored at the corner index that is lower in
// a = C+1 and b = C+2)
// ---------------------------------------------------------------------------

// The face fluxes of every active direction and the edge EMFs the flux tasks do not
// write, in one launch (resistive UCT, FP64 or mixed precision).  Block ranges select
// the task (the same items, march lengths and grid copies as separate launches would
// take, so every face and edge is bitwise the same); one launch keeps the SMs filled
// across what would be three to six single-wave kernels with their tails.
template <typename T>
struct StencilTasks {
    int b0[7];                 // first block of task s (flux x, y, z; EMF x, y, z); b0[6] = grid
    int emarch[3];             // EMF task C marches along C + 2 (both transverse directions active)
    Dims g[6];                 // each task's copy of the grid, with its march length
    FluxArgs<T> fa[3];
    EmfArgs<T> ea[3];
};

#ifdef GRMHD_STENCIL_INSTANCE
// threads per block of an instance
template <typename T, bool P>
constexpr int stencil_threads()
{
    return sizeof(T) == 8 ? Flux64<P, false>::NT : 128;
}

// the flux task along d (FP32: d = D)
template <int D, bool M, typename T, bool P>
__device__ __forceinline__ void stencil_flux(const Dims& g, int d, const FluxArgs<T>& a, long long t0, long long nt,
                                             double* sm)
{
    const long long tot = g.dq[d].d * (d == 0 ? (long long)g.n[1] * g.n[2]
                                              : (d == 1 ? (long long)g.n[0] * g.n[2] : (long long)g.n[0] * g.n[1]));
    for (long long t = t0; t < tot; t += nt) {
        if constexpr (sizeof(T) == 8)
            flux64_item<M, P, false>(g, d, a.prim.p, a.bf.p, nullptr, a.psi, a.alp, a.F.p, nullptr, a.Eh, sm, t);
        else flux32_item<D, M, P>(g, a.prim, a.bf, a.psi, a.alp, a.F, a.Eh, t);
    }
}

// one edge per thread (an edge direction with one inactive transverse direction)
template <int C, bool M, typename T, bool P>
__device__ __forceinline__ void stencil_emf_single(const Dims& g, const EmfArgs<T>& a, long long t0, long long nt)
{
    long long tot = 1;
#pragma unroll
    for (int d = 0; d < 3; d++) tot *= (d == C) ? g.n[d] : (g.act[d] ? g.n[d] + 1 : 1);
    for (long long t = t0; t < tot; t += nt) emf_item<C, M, T, P>(g, a.prim, a.bf, a.psi, a.alp, a.Eh, t);
}

// marched edges of direction c
template <bool M, typename T, bool P>
__device__ __forceinline__ void stencil_emf_march(const Dims& g, int c, const EmfArgs<T>& a, long long t0, long long nt)
{
    const int A = c == 2 ? 0 : c + 1, B = c == 0 ? 2 : c - 1;
    const long long tot = (long long)g.dq[B].d * g.n[c] * (g.n[A] + 1);
    for (long long t = t0; t < tot; t += nt) emf_line_item<M, T, P>(g, c, a.prim.p, a.bf.p, a.psi, a.alp, a.Eh, t);
}

// The FP32 PPM instance is held to 96 registers (five blocks per SM, 160 B of spills):
// at its natural 128 it ran 2 % slower.  The others keep the compiler's choice.
template <bool M, typename T, bool P>
__global__ void __launch_bounds__(stencil_threads<T, P>(), sizeof(T) == 8 ? (P ? 6 : 4) : (P ? 5 : 0)) k_stencil(StencilTasks<T> L)
{
    __shared__ double sm[sizeof(T) == 8 ? Flux64<P, false>::SM : 1];
    grid_dep_sync();
    const int b = blockIdx.x;
    int s = 0;
#pragma unroll
    for (int i = 1; i < 6; i++)
        if (b >= L.b0[i]) s = i;   // empty tasks have b0[i] == b0[i + 1]
    const long long nt = (long long)(L.b0[s + 1] - L.b0[s]) * blockDim.x;
    const long long t0 = (long long)(b - L.b0[s]) * blockDim.x + threadIdx.x;
    // the FP64 fluxes and the marched edges take the direction as a run-time value: one code
    if constexpr (sizeof(T) == 8) {
        if (s < 3) {
            stencil_flux<0, M, T, P>(L.g[s], s, L.fa[s], t0, nt, sm);
            return;
        }
    }
    if (s >= 3 && L.emarch[s - 3]) {
        stencil_emf_march<M, T, P>(L.g[s], s - 3, L.ea[s - 3], t0, nt);
        return;
    }
    switch (s) {
#define GRMHD_STENCIL_EMF(C)                                                                       \
    case 3 + C: stencil_emf_single<C, M, T, P>(L.g[3 + C], L.ea[C], t0, nt); break;
#define GRMHD_STENCIL_FLUX(D)                                                                      \
    case D:                                                                                        \
        if constexpr (sizeof(T) == 4) stencil_flux<D, M, T, P>(L.g[D], D, L.fa[D], t0, nt, sm);    \
        break;
        GRMHD_STENCIL_FLUX(0)
        GRMHD_STENCIL_FLUX(1)
        GRMHD_STENCIL_FLUX(2)
        GRMHD_STENCIL_EMF(0)
        GRMHD_STENCIL_EMF(1)
        GRMHD_STENCIL_EMF(2)
#undef GRMHD_STENCIL_EMF
#undef GRMHD_STENCIL_FLUX
    default: break;
    }
}

#endif

// the launch of one instance: march lengths and block ranges of every task
template <bool M, typename T, bool P>
cudaError_t stencil_launch(const Dims& g, const PrimIn<T>& prim, CP3 bf, const double* psi, const double* alp,
                           const FluxOut<T>* F, double* const (*fe)[3], double* const* Eh, int nsm, cudaStream_t st)
#ifdef GRMHD_STENCIL_INSTANCE
{
    constexpr int NT = stencil_threads<T, P>();
    static int nb_sm = 0;   // resident blocks per SM, queried once
    if (nb_sm < 1) {
        int q = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, k_stencil<M, T, P>, NT, 0) != cudaSuccess || q < 1)
            q = 1;
        nb_sm = q;
    }
    const int bps = nb_sm;
    const double c0 = sizeof(T) == 8 ? Flux64<P, false>::C0 : (P ? 1.0 : 0.6);
    StencilTasks<T> L;
    memset(&L, 0, sizeof L);
    int nb = 0;
    for (int d = 0; d < 3; d++) {
        L.b0[d] = nb;
        L.g[d] = g;
        FluxArgs<T>& a = L.fa[d];
        a.prim = prim;
        a.bf = bf;
        a.psi = psi;
        a.alp = alp;
        if (!g.act[d]) continue;
        a.F = F[d];
        for (int k = 0; k < 3; k++) a.Eh[k] = fe && !M ? fe[d][k] : nullptr;
        const long long other = d == 0 ? (long long)g.n[1] * g.n[2]
                                       : (d == 1 ? (long long)g.n[0] * g.n[2] : (long long)g.n[0] * g.n[1]);
        set_march(L.g[d], d, march_len(g.n[d], other, nsm, bps, c0, NT));
        nb += grid_for((long long)L.g[d].dq[d].d * other, NT, nsm);
    }
    for (int c = 0; c < 3; c++) {
        L.b0[3 + c] = nb;
        L.g[3 + c] = g;
        EmfArgs<T>& a = L.ea[c];
        a.prim = prim;
        a.bf = bf;
        a.psi = psi;
        a.alp = alp;
        if (!Eh || !Eh[c]) continue;
        a.Eh = Eh[c];
        const int A = (c + 1) % 3, B = (c + 2) % 3;
        if (g.act[A] && g.act[B]) {
            const long long other = (long long)g.n[c] * (g.n[A] + 1);
            set_march(L.g[3 + c], B, march_len(g.n[B], other, nsm, bps, c0, NT));
            L.emarch[c] = 1;
            nb += grid_for((long long)L.g[3 + c].dq[B].d * other, NT, nsm);
        } else {
            nb += grid_for(emf_work(g, c), NT, nsm);
        }
    }
    L.b0[6] = nb;
    if (nb == 0) return cudaSuccess;
    launch_k(k_stencil<M, T, P>, nb, NT, st, L);
    return cudaGetLastError();
}
#else
;
#endif

}  // namespace grmhd
