// GLM hyperbolic divergence cleaning (arXiv 2110.03732 Sec. 3.1) with cell-centred
// magnetic fields: the explicit part of an IMEX stage for 12 cell-centred variables
// (D, S_1..3, tau, E^1..3, q_B^1..3, q_Phi), sm_103a, FP64.
//
//   k_glm_flux    MC reconstruction of the 8 primitives, B^i = q_B^i/psi^6 and
//                  Phi = q_Phi/psi^6 to the D-faces; HLL flux of all 12 with the
//                  maximal-diffusivity speeds of Sec. 2.5.  With beta = 0:
//                    (f_B^j)^D = eta^{jDk} alpha E_k,   (f_Phi)^D = alpha q_B^D
//   k_glm_update   flux divergence + sources: the Gauss-law charge term of s_E and the
//                  metric terms of s_S, s_tau (Sec. 2.1), and for the new fields
//                    s_B^i  = -psi^6 alpha gamma^{ij} d_j Phi = -alpha psi^2 d_i Phi
//                    s_Phi  = -alpha kappa_B q_Phi + q_B^i d_i alpha
//                  (central differences of cell values); writes L, or folds it into the
//                  IMEX stage bases and the final combination (Sec. 2.3)
//
// Phi's flux divergence enters with the sign of the conservative form of Sec. 2.1
// (d_t q + d_i f^i = s with the f_Phi and s_Phi of Sec. 3.1), which makes (B, Phi) a
// damped wave system.  The charge field Psi is not evolved; rho_e comes from Gauss's
// law as in the staggered scheme.  The implicit solve is the one of Sec. 2.4 with the
// cell-centred field (k_implicit_cc in implicit.cu).
#include "grmhd_device.cuh"
#include "items.cuh"
#include "kernels.h"
#include "launch.cuh"

namespace grmhd {

// The fluxes of every active direction in one launch (block ranges select the direction, as
// the tasks of k_stencil): the launches per direction were single-wave, and their tails left
// SMs idle (384^2: 2 x 41 us, 73.5 us in one launch).
struct GlmTasks {
    int b0[4];    // first block of direction d; b0[3] = grid
    Dims g[3];    // each direction's copy of the grid, with its march length
    GlmFluxArgs a;
};

template <bool M, bool P>
__global__ void __launch_bounds__(Flux64<P, true>::NT, P ? 6 : 4) k_glm_flux(const __grid_constant__ GlmTasks L)
{
    __shared__ double sm[Flux64<P, true>::SM];
    grid_dep_sync();
    const int b = blockIdx.x;
    const int d = b >= L.b0[2] ? 2 : (b >= L.b0[1] ? 1 : 0);   // empty directions have b0[d] == b0[d + 1]
    const Dims& g = L.g[d];
    const long long nt = (long long)(L.b0[d + 1] - L.b0[d]) * blockDim.x;
    const long long tot = g.dq[d].d * (d == 0 ? (long long)g.n[1] * g.n[2]
                                              : (d == 1 ? (long long)g.n[0] * g.n[2] : (long long)g.n[0] * g.n[1]));
    for (long long t = (long long)(b - L.b0[d]) * blockDim.x + threadIdx.x; t < tot; t += nt)
        flux64_item<M, P, true>(g, d, L.a.prim, L.a.qB, L.a.qphi, L.a.psi, L.a.alp, L.a.F[d], nullptr, nullptr, sm, t);
}

__device__ __forceinline__ void glm_out(const GlmUpdateArgs& a, int v, long long o, double L, bool has_r)
{
    if (a.mode == UPD_WRITE_L) {
        a.L[v][o] = L;
        return;
    }
    // as out_value: host-formed dt products, q^n read at stage 0 only
    const double r = has_r ? a.R[v - 5][o] : 0.0;
    const double qn = a.stage == 0 ? a.qn[v][o] : 0.0;
    for (int k = a.stage + 1; k < a.s; k++) {
        const double prev = a.stage == 0 ? qn : a.base[k][v][o];
        double nb = prev + a.cL[k] * L;
        if (has_r) nb += a.cR[k] * r;
        a.base[k][v][o] = nb;
    }
    const double prev = a.stage == 0 ? qn : a.acc[v][o];
    double nv = prev + a.cwL * L;
    if (has_r) nv += a.cwR * r;
    if (a.stage == a.s - 1) a.qn[v][o] = nv;
    else a.acc[v][o] = nv;
}

template <bool M>
__device__ __forceinline__ void glm_update_item(const Dims& g, const GlmUpdateArgs& a, long long t)
{
    const double* __restrict__ psi = M ? a.psi : nullptr;
    const double* __restrict__ alp = M ? a.alp : nullptr;
    int c[3];
    interior_coords(g, t, c);
    const long long o = lin(g, c[0], c[1], c[2]);
    double Lc[12];
    cell_sources<M, true>(g, a.prim, a.qB, nullptr, psi, alp, c, o, Lc);
#pragma unroll
    for (int v = 0; v < 12; v++)
        if (v == 0 || v >= 8 || (!M && v < 5)) Lc[v] = 0.0;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        if (!g.act[d]) continue;
        const long long o1 = chk(g, o + g.st[d]);
        const double hidx = 0.5 * g.idx[d];   // F holds twice the flux
#pragma unroll
        for (int v = 0; v < 12; v++) {
            const double* __restrict__ Fv = a.F[d][v];
            Lc[v] -= (Fv[o1] - Fv[o]) * hidx;
        }
    }
    const double ps = psi ? psi[o] : 1.0;
    const double al = alp ? alp[o] : 1.0;
    const double p2 = ps * ps;
    Lc[11] -= al * a.kappa * a.qphi[o];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        if (!g.act[d]) continue;
        int cp[3] = {c[0], c[1], c[2]}, cm[3] = {c[0], c[1], c[2]};
        cp[d] += 1;
        cm[d] -= 1;
        double sp = psi ? psi[chk(g, o + g.st[d])] : 1.0, sm = psi ? psi[chk(g, o - g.st[d])] : 1.0;
        sp = sp * sp;
        sm = sm * sm;
        const double sp3 = sp * sp * sp, sm3 = sm * sm * sm, r = rcp_pos(sp3 * sm3);
        const double php = a.qphi[cell_at(g, cp)] * (sm3 * r);   // q_Phi / psi^6
        const double phm = a.qphi[cell_at(g, cm)] * (sp3 * r);
        Lc[8 + d] -= al * p2 * ((php - phm) * (0.5 * g.idx[d]));
        if (alp) Lc[11] += a.qB[d][o] * ((alp[chk(g, o + g.st[d])] - alp[chk(g, o - g.st[d])]) * (0.5 * g.idx[d]));
    }
#pragma unroll
    for (int v = 0; v < 12; v++) glm_out(a, v, o, Lc[v], v >= 5 && v < 8);
}

__global__ void __launch_bounds__(128) k_glm_update_flat(Dims g, GlmUpdateArgs a)
{
    grid_dep_sync();
    const long long tot = (long long)g.n[0] * g.n[1] * g.n[2];
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x)
        glm_update_item<false>(g, a, t);
}

__global__ void __launch_bounds__(128) k_glm_update_metric(Dims g, GlmUpdateArgs a)
{
    grid_dep_sync();
    const long long tot = (long long)g.n[0] * g.n[1] * g.n[2];
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x)
        glm_update_item<true>(g, a, t);
}

// faces per thread as for the staggered-field flux kernels
template <bool M, bool P>
static cudaError_t glm_flux_launch(const Dims& g, const GlmFluxArgs& a, int nsm, cudaStream_t st)
{
    constexpr int NT = Flux64<P, true>::NT;
    static int nb_sm = 0;   // resident blocks per SM, queried once
    if (nb_sm < 1) {
        int q = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, k_glm_flux<M, P>, NT, 0) != cudaSuccess || q < 1) q = 1;
        nb_sm = q;
    }
    GlmTasks L;
    L.a = a;
    int nb = 0;
    for (int d = 0; d < 3; d++) {
        L.b0[d] = nb;
        L.g[d] = g;
        if (!g.act[d]) continue;
        const long long other = d == 0 ? (long long)g.n[1] * g.n[2]
                                       : (d == 1 ? (long long)g.n[0] * g.n[2] : (long long)g.n[0] * g.n[1]);
        set_march(L.g[d], d, march_len(g.n[d], other, nsm, nb_sm, Flux64<P, true>::C0, NT));
        nb += grid_for((long long)L.g[d].dq[d].d * other, NT, nsm);
    }
    L.b0[3] = nb;
    launch_k(k_glm_flux<M, P>, nb, NT, st, L);
    return cudaGetLastError();
}

cudaError_t launch_glm_flux(const Dims& g, const GlmFluxArgs& a, int nsm, cudaStream_t st, bool ppm)
{
    const bool m = a.psi || a.alp;
    if (ppm) return m ? glm_flux_launch<true, true>(g, a, nsm, st) : glm_flux_launch<false, true>(g, a, nsm, st);
    return m ? glm_flux_launch<true, false>(g, a, nsm, st) : glm_flux_launch<false, false>(g, a, nsm, st);
}

cudaError_t launch_glm_update(const Dims& g, const GlmUpdateArgs& a, int nsm, cudaStream_t st)
{
    const int b = grid_for((long long)g.n[0] * g.n[1] * g.n[2], 128, nsm);
    launch_k(a.psi || a.alp ? k_glm_update_metric : k_glm_update_flat, b, 128, st, g, a);
    return cudaGetLastError();
}

GRMHD_OOB_READER(oob_glm)

}  // namespace grmhd
