// Face fluxes in launches of their own, FP64: the one flux direction of a flat 1-D grid,
// and the fluxes (which also write the transport velocities) and edge EMFs of the
// ideal-limit variant (App. A).  Every other stage takes k_stencil (stencil.cuh).
#include "grmhd_device.cuh"
#include "items.cuh"
#include "kernels.h"
#include "launch.cuh"

namespace grmhd {

// MC (or PPM) fluxes, K consecutive D-faces per thread (flux64_item)
template <int D, bool M, bool P = false>
__global__ void __launch_bounds__(Flux64<P, false>::NT, 4) k_flux_march(Dims g, FluxArgs<double> a)
{
    __shared__ double sm[Flux64<P, false>::SM];
    grid_dep_sync();
    const long long nq = g.dq[D].d;   // chunks of g.mk[D] faces per line
    const long long tot = nq * (D == 0 ? (long long)g.n[1] * g.n[2]
                                       : (D == 1 ? (long long)g.n[0] * g.n[2] : (long long)g.n[0] * g.n[1]));
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x)
        flux64_item<M, P, false>(g, D, a.prim.p, a.bf.p, nullptr, a.psi, a.alp, a.F.p, a.vbar, a.Eh, sm, t);
}

// ideal-limit edge EMF (App. A) from the stored transport velocities
struct VbarArgs {
    const double* p[3][2];
};

template <int C, bool M>
__global__ void __launch_bounds__(128) k_emf_ideal(Dims g, EmfArgs<double> a, VbarArgs vb)
{
    grid_dep_sync();
    long long tot = 1;
#pragma unroll
    for (int d = 0; d < 3; d++) tot *= (d == C) ? g.n[d] : (g.act[d] ? g.n[d] + 1 : 1);
    CP8 prim;
#pragma unroll
    for (int v = 0; v < 8; v++) prim.p[v] = a.prim.p[v];
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x)
        emf_ideal_item<C, M>(g, prim, a.bf, a.psi, a.alp, vb.p, a.Eh, t);
}

// faces per thread by march_len
template <int D, bool M, bool P>
static void flux_march_launch(const Dims& g, int nsm, cudaStream_t st, const FluxArgs<double>& a)
{
    constexpr int NT = Flux64<P, false>::NT;
    const long long other = D == 0 ? (long long)g.n[1] * g.n[2]
                                   : (D == 1 ? (long long)g.n[0] * g.n[2] : (long long)g.n[0] * g.n[1]);
    static int nb_sm = 0;   // resident blocks per SM, queried once
    if (nb_sm < 1) {
        int q = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, k_flux_march<D, M, P>, NT, 0) != cudaSuccess || q < 1)
            q = 1;
        nb_sm = q;
    }
    const int K = march_len(g.n[D], other, nsm, nb_sm, Flux64<P, false>::C0, NT);
    Dims gl = g;
    set_march(gl, D, K);
    launch_k(k_flux_march<D, M, P>, grid_for((long long)gl.dq[D].d * other, NT, nsm), NT, st, gl, a);
}

static void flux_dispatch(const Dims& g, int d, bool m, int nsm, cudaStream_t st, const FluxArgs<double>& a)
{
    if (d == 0) m ? flux_march_launch<0, true, false>(g, nsm, st, a) : flux_march_launch<0, false, false>(g, nsm, st, a);
    else if (d == 1) m ? flux_march_launch<1, true, false>(g, nsm, st, a) : flux_march_launch<1, false, false>(g, nsm, st, a);
    else m ? flux_march_launch<2, true, false>(g, nsm, st, a) : flux_march_launch<2, false, false>(g, nsm, st, a);
}

cudaError_t launch_flux(const Dims& g, int d, CP8 prim, CP3 bf, const double* psi, const double* alp, P8 F, int nsm,
                        cudaStream_t st, double* const* vbar, bool ppm, double* const* Eh)
{
    FluxArgs<double> a;
    for (int k = 0; k < 3; k++) a.Eh[k] = Eh && !(psi || alp) ? Eh[k] : nullptr;
    for (int v = 0; v < 8; v++) {
        a.prim.p[v] = prim.p[v];
        a.F.p[v] = F.p[v];
    }
    a.vbar[0] = vbar ? vbar[0] : nullptr;
    a.vbar[1] = vbar ? vbar[1] : nullptr;
    a.bf = bf;
    a.psi = psi;
    a.alp = alp;
    // PPM comes here on flat 1-D grids only (it does not take the ideal-limit EMF)
    if (ppm) flux_march_launch<0, false, true>(g, nsm, st, a);
    else flux_dispatch(g, d, psi || alp, nsm, st, a);
    return cudaGetLastError();
}

cudaError_t launch_emf_ideal(const Dims& g, int c, CP8 prim, CP3 bf, const double* psi, const double* alp,
                             const double* const (*vb)[2], double* Eh, int nsm, cudaStream_t st)
{
    EmfArgs<double> a;
    for (int v = 0; v < 8; v++) a.prim.p[v] = prim.p[v];
    a.bf = bf;
    a.psi = psi;
    a.alp = alp;
    a.Eh = Eh;
    VbarArgs v;
    for (int d = 0; d < 3; d++)
        for (int k = 0; k < 2; k++) v.p[d][k] = vb[d][k];
    const int b = grid_for(emf_work(g, c), 128, nsm);
    const bool m = psi || alp;
    if (c == 0) launch_k(m ? k_emf_ideal<0, true> : k_emf_ideal<0, false>, b, 128, st, g, a, v);
    else if (c == 1) launch_k(m ? k_emf_ideal<1, true> : k_emf_ideal<1, false>, b, 128, st, g, a, v);
    else launch_k(m ? k_emf_ideal<2, true> : k_emf_ideal<2, false>, b, 128, st, g, a, v);
    return cudaGetLastError();
}

GRMHD_OOB_READER(oob_flux)

}  // namespace grmhd
