// CUDA kernels of one IMEX-RK stage of resistive (GR)MHD with staggered
// constrained transport (arXiv 2110.03732), sm_103a, FP64 and mixed precision.
//
// In this file: the update, the set-up kernels and the reductions.  The others:
//   k_implicit (implicit.cu)  Sec. 2.4: per-cell Newton on u coupled to the implicit E update;
//                writes stage primitives and the stiff rate R = (q_E - q_E,base)/(a_ii dt)
//   k_stencil<M, T, P> (stencil.cuh)  one launch per stage of
//                - the flux tasks, Sec. 2.1 + Sec. 5 defaults: MC (or PPM)
//                  reconstruction to the D-faces, marched along D, and the HLL flux with
//                  the maximal-diffusivity speeds of Sec. 2.5 (on flat 1-D / 2-D grids
//                  also the degenerate edge EMFs), and
//                - the edge-EMF tasks, Sec. 3.2 steps (i)-(vii): the upwind (UCT-HLL)
//                  edge EMF hat{E}_C, marched along C + 2 when both transverse
//                  directions are active
//                in FP64 or (T = float) mixed precision
//   k_flux_march<D>, k_emf_ideal<C> (flux.cu)  the fluxes and App. A edge EMF of the ideal-limit
//                variant (separate launches: the flux writes the transport velocities)
//   k_update<M>  flux divergence + non-stiff sources (Sec. 2.1) and the CT face update
//                (Sec. 3.2); writes L, or folds it straight into the IMEX stage bases and
//                the final combination (Sec. 2.3)
//   k_prim2con, k_curlA (Sec. 4), k_dt (Sec. 2.5), k_divb, k_totals: set-up and
//   diagnostics; k_curlA_cc, k_prim2con_cc, k_diag_cc: the same for the cell-centred fields
//   of the GLM variant (its flux and update kernels: glm.cu; k_implicit_cc: implicit.cu)
#include "grmhd_device.cuh"
#include "items.cuh"
#include "kernels.h"
#include "launch.cuh"
#include "stencil.cuh"

namespace grmhd {

thread_local bool launch_overlap = false;

// ---------------------------------------------------------------------------
// update: cell-centred L (flux divergence + non-stiff sources) and face L_B (CT)
// ---------------------------------------------------------------------------

// Register bounds, us per launch.  The FP32-flux instances take 32 registers (16 blocks per
// SM; one variable at a time, 90-240 B of spills): 512^2 40.0 against 46.4 at 8 to 12 blocks,
// 96^3 star 166 against 199-214 (42 and 181 with all eight divergences held at once).  FP64:
// seven blocks flat (512^2 55.7; 56.5 unbounded, 58.2 at eight), ten with a metric (128^3
// 748; 778 at twelve, 760 at eight; 903 before the sources were collected; at ten it is 756 with
// the trace of the sources summed from its positive terms).
//
// A grid that fits five blocks per SM waits for each variable's loads in turn, not for
// registers: there the FP32-flux instances hold all eight divergences at once (96 registers,
// ALL in update_item).  us per launch, one variable at a time / all at once: star 24^3 27.3 /
// 24.9, 40^3 30.2 / 27.3, vortex 224^2 20.9 / 19.1, 96^2 19.9 / 19.5; 48^3 (5.7 blocks) 34.6 either
// way.
constexpr int kUpdateSmall = 5;   // blocks per SM of the ALL instances (launch_update)

template <bool M, bool F32, bool ALL = false>
__global__ void __launch_bounds__(128, ALL ? kUpdateSmall : (F32 ? 16 : (M ? 10 : 7))) k_update(Dims g, UpdateArgs a)
{
    grid_dep_sync();
    long long tot = 1;
#pragma unroll
    for (int d = 0; d < 3; d++) tot *= g.act[d] ? g.n[d] + 1 : 1;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x)
        update_item<M, F32, ALL>(g, a, t);
}

// ---------------------------------------------------------------------------
// set-up: face q_B = curl of the edge potential (Sec. 4), prim -> cons (Sec. 2.1)
// ---------------------------------------------------------------------------

__global__ void k_curlA(Dims g, CP3 A, P3 bf)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < g.ncell;
         t += (long long)gridDim.x * blockDim.x) {
        int c[3];
        c[0] = (int)(t % g.N[0]);
        c[1] = (int)((t / g.N[0]) % g.N[1]);
        c[2] = (int)(t / ((long long)g.N[0] * g.N[1]));
#pragma unroll
        for (int fa = 0; fa < 3; fa++) {
            const int fb = (fa + 1) % 3, fc = (fa + 2) % 3;
            if ((g.act[fb] && c[fb] + 1 >= g.N[fb]) || (g.act[fc] && c[fc] + 1 >= g.N[fc])) continue;
            double r = 0.0;
            if (g.act[fb]) r += (A.p[fc][chk(g, t + g.st[fb])] - A.p[fc][t]) * g.idx[fb];
            if (g.act[fc]) r -= (A.p[fb][chk(g, t + g.st[fc])] - A.p[fb][t]) * g.idx[fc];
            bf.p[fa][t] = r;
        }
    }
}

__global__ void k_prim2con(Dims g, CP8 prim, CP3 bf, const double* __restrict__ psi, P8 q)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < g.ncell;
         t += (long long)gridDim.x * blockDim.x) {
        int c[3];
        c[0] = (int)(t % g.N[0]);
        c[1] = (int)((t / g.N[0]) % g.N[1]);
        c[2] = (int)(t / ((long long)g.N[0] * g.N[1]));
        const double ps = psi ? psi[t] : 1.0;
        const double p2 = ps * ps, p6 = p2 * p2 * p2;
        double pr[8], B[3];
#pragma unroll
        for (int v = 0; v < 8; v++) pr[v] = prim.p[v][t];
#pragma unroll
        for (int e = 0; e < 3; e++) B[e] = cell_qB(g, bf.p[e], e, c) / p6;
        FaceState s;
        face_state(pr, B, 0, ps, 1.0, g.gh, s);
#pragma unroll
        for (int v = 0; v < 8; v++) q.p[v][t] = s.q[v];
    }
}

// cell-centred q_B^i = eta^{ijk} d_j A_k from a cell-centred potential by central
// differences (Sec. 4, cell-centred fields), interior cells; the potential is read
// as given on the whole padded grid
__global__ void k_curlA_cc(Dims g, CP3 A, P3 qB)
{
    const long long tot = (long long)g.n[0] * g.n[1] * g.n[2];
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x) {
        const int i = g.ng[0] + (int)(t % g.n[0]);
        const int j = g.ng[1] + (int)((t / g.n[0]) % g.n[1]);
        const int k = g.ng[2] + (int)(t / ((long long)g.n[0] * g.n[1]));
        const long long o = lin(g, i, j, k);
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int b = (a + 1) % 3, c = (a + 2) % 3;
            double r = 0.0;
            if (g.act[b]) r += (A.p[c][chk(g, o + g.st[b])] - A.p[c][chk(g, o - g.st[b])]) * (0.5 * g.idx[b]);
            if (g.act[c]) r -= (A.p[b][chk(g, o + g.st[c])] - A.p[b][chk(g, o - g.st[c])]) * (0.5 * g.idx[c]);
            qB.p[a][o] = r;
        }
    }
}

// prim -> cons with cell-centred q_B, every padded cell; q_Phi = psi^6 Phi (Sec. 3.1)
// from the primitive Phi (NULL: zero)
__global__ void k_prim2con_cc(Dims g, CP8 prim, CP3 qB, const double* __restrict__ psi,
                              const double* __restrict__ phi, double* __restrict__ qphi, P8 q)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < g.ncell;
         t += (long long)gridDim.x * blockDim.x) {
        const double ps = psi ? psi[t] : 1.0;
        const double p2 = ps * ps, p6 = p2 * p2 * p2;
        double pr[8], B[3];
#pragma unroll
        for (int v = 0; v < 8; v++) pr[v] = prim.p[v][t];
#pragma unroll
        for (int e = 0; e < 3; e++) B[e] = qB.p[e][t] / p6;
        FaceState s;
        face_state(pr, B, 0, ps, 1.0, g.gh, s);
#pragma unroll
        for (int v = 0; v < 8; v++) q.p[v][t] = s.q[v];
        qphi[t] = phi ? p6 * phi[t] : 0.0;
    }
}

// FP32 copy of caller primitives at every padded cell (fixed-boundary ghosts
// included) with the densitised cell-centred q_B, for the mixed-precision path
__global__ void k_prim_to32(Dims g, CP8 prim, CP3 bf, F11 p32)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < g.ncell;
         t += (long long)gridDim.x * blockDim.x) {
        int c[3];
        c[0] = (int)(t % g.N[0]);
        c[1] = (int)((t / g.N[0]) % g.N[1]);
        c[2] = (int)(t / ((long long)g.N[0] * g.N[1]));
#pragma unroll
        for (int v = 0; v < 8; v++) p32.p[v][t] = (float)prim.p[v][t];
#pragma unroll
        for (int e = 0; e < 3; e++) p32.p[8 + e][t] = (float)cell_qB(g, bf.p[e], e, c);
    }
}

// ---------------------------------------------------------------------------
// reductions (fixed-order block trees: deterministic for a given launch shape)
// ---------------------------------------------------------------------------

template <typename Op>
__device__ __forceinline__ double block_reduce(double v, Op op, double* sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_down_sync(0xffffffffu, v, o));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    const int nw = blockDim.x >> 5;
    if (w == 0) {
        v = l < nw ? sh[l] : 0.0;   // identity of sum, and of max over non-negative values
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_down_sync(0xffffffffu, v, o));
    }
    __syncthreads();
    return v;
}

struct OpSum { __device__ double operator()(double a, double b) const { return a + b; } };
struct OpMax { __device__ double operator()(double a, double b) const { return fmax(a, b); } };

// per block: [max over cells of sum_d alpha sqrt(gamma^dd)/dx_d]
__global__ void __launch_bounds__(256) k_dt(Dims g, const double* __restrict__ psi, const double* __restrict__ alp,
                                            double* __restrict__ part)
{
    __shared__ double sh[32];
    const long long tot = (long long)g.n[0] * g.n[1] * g.n[2];
    double m = 0.0;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x) {
        const int i = g.ng[0] + (int)(t % g.n[0]);
        const int j = g.ng[1] + (int)((t / g.n[0]) % g.n[1]);
        const int k = g.ng[2] + (int)(t / ((long long)g.n[0] * g.n[1]));
        const long long o = lin(g, i, j, k);
        const double ps = psi ? psi[o] : 1.0;
        const double sp = (alp ? alp[o] : 1.0) / (ps * ps);
        m = fmax(m, sp * (g.idx[0] + g.idx[1] + g.idx[2]));
    }
    m = block_reduce(m, OpMax(), sh);
    if (threadIdx.x == 0) part[blockIdx.x] = m;
}

// per block: [sum |div q_B|, sum div^2, max |div|, sum q_0..q_7 (times dV)]
__global__ void __launch_bounds__(256) k_diag(Dims g, CP3 bf, CP8 q, double dV, double* __restrict__ part)
{
    __shared__ double sh[32];
    const long long tot = (long long)g.n[0] * g.n[1] * g.n[2];
    double s1 = 0.0, s2 = 0.0, mx = 0.0, tq[8];
#pragma unroll
    for (int v = 0; v < 8; v++) tq[v] = 0.0;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x) {
        int c[3];
        c[0] = g.ng[0] + (int)(t % g.n[0]);
        c[1] = g.ng[1] + (int)((t / g.n[0]) % g.n[1]);
        c[2] = g.ng[2] + (int)(t / ((long long)g.n[0] * g.n[1]));
        const long long o = lin(g, c[0], c[1], c[2]);
        const double dv = cell_divb(g, bf.p, c, o);
        s1 += fabs(dv);
        s2 += dv * dv;
        mx = fmax(mx, fabs(dv));
#pragma unroll
        for (int v = 0; v < 8; v++) tq[v] += q.p[v][o] * dV;
    }
    double r = block_reduce(s1, OpSum(), sh);
    if (threadIdx.x == 0) part[blockIdx.x * 11 + 0] = r;
    r = block_reduce(s2, OpSum(), sh);
    if (threadIdx.x == 0) part[blockIdx.x * 11 + 1] = r;
    r = block_reduce(mx, OpMax(), sh);
    if (threadIdx.x == 0) part[blockIdx.x * 11 + 2] = r;
#pragma unroll
    for (int v = 0; v < 8; v++) {
        r = block_reduce(tq[v], OpSum(), sh);
        if (threadIdx.x == 0) part[blockIdx.x * 11 + 3 + v] = r;
    }
}

// the same with cell-centred q_B: div by central differences (GLM variant)
__global__ void __launch_bounds__(256) k_diag_cc(Dims g, CP3 qB, CP8 q, double dV, double* __restrict__ part)
{
    __shared__ double sh[32];
    const long long tot = (long long)g.n[0] * g.n[1] * g.n[2];
    double s1 = 0.0, s2 = 0.0, mx = 0.0, tq[8];
#pragma unroll
    for (int v = 0; v < 8; v++) tq[v] = 0.0;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x) {
        int c[3];
        c[0] = g.ng[0] + (int)(t % g.n[0]);
        c[1] = g.ng[1] + (int)((t / g.n[0]) % g.n[1]);
        c[2] = g.ng[2] + (int)(t / ((long long)g.n[0] * g.n[1]));
        const long long o = lin(g, c[0], c[1], c[2]);
        double dv = 0.0;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            if (!g.act[d]) continue;
            int cu[3] = {c[0], c[1], c[2]}, cl[3] = {c[0], c[1], c[2]};
            cu[d] += 1;
            cl[d] -= 1;
            dv += (qB.p[d][cell_at(g, cu)] - qB.p[d][cell_at(g, cl)]) * (0.5 * g.idx[d]);
        }
        s1 += fabs(dv);
        s2 += dv * dv;
        mx = fmax(mx, fabs(dv));
#pragma unroll
        for (int v = 0; v < 8; v++) tq[v] += q.p[v][o] * dV;
    }
    double r = block_reduce(s1, OpSum(), sh);
    if (threadIdx.x == 0) part[blockIdx.x * 11 + 0] = r;
    r = block_reduce(s2, OpSum(), sh);
    if (threadIdx.x == 0) part[blockIdx.x * 11 + 1] = r;
    r = block_reduce(mx, OpMax(), sh);
    if (threadIdx.x == 0) part[blockIdx.x * 11 + 2] = r;
#pragma unroll
    for (int v = 0; v < 8; v++) {
        r = block_reduce(tq[v], OpSum(), sh);
        if (threadIdx.x == 0) part[blockIdx.x * 11 + 3 + v] = r;
    }
}

// second pass: one block folds `nb` partial rows of width `w`; column kinds: 0 sum, 1 max
__global__ void __launch_bounds__(256) k_fold(const double* __restrict__ part, int nb, int w,
                                              const int* __restrict__ kinds_unused, unsigned kinds_mask,
                                              double* __restrict__ out)
{
    __shared__ double sh[32];
    (void)kinds_unused;
    for (int col = 0; col < w; col++) {
        const bool is_max = (kinds_mask >> col) & 1u;
        double v = 0.0;
        for (int b = threadIdx.x; b < nb; b += blockDim.x) {
            const double x = part[(long long)b * w + col];
            v = is_max ? fmax(v, x) : v + x;
        }
        v = is_max ? block_reduce(v, OpMax(), sh) : block_reduce(v, OpSum(), sh);
        if (threadIdx.x == 0) out[col] = v;
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(256) k_hist_init(long long n, const double* __restrict__ u1,
                                                   const double* __restrict__ u2, const double* __restrict__ u3,
                                                   const double* __restrict__ psi, P3f hs, P3f hd)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        const double p2 = psi ? psi[t] * psi[t] : 1.0;
        hs.p[0][t] = (float)(p2 * u1[t]);
        hs.p[1][t] = (float)(p2 * u2[t]);
        hs.p[2][t] = (float)(p2 * u3[t]);
        hd.p[0][t] = hd.p[1][t] = hd.p[2][t] = 0.0f;
    }
}

cudaError_t launch_hist_init(const Dims& g, const double* u1, const double* u2, const double* u3, const double* psi,
                             P3f hs, P3f hd, int nsm, cudaStream_t st)
{
    k_hist_init<<<grid_for(g.ncell, 256, nsm), 256, 0, st>>>(g.ncell, u1, u2, u3, psi, hs, hd);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t stencil_dispatch(const Dims& g, const PrimIn<T>& prim, CP3 bf, const double* psi, const double* alp,
                                    const FluxOut<T>* F, double* const (*fe)[3], double* const* Eh, int nsm,
                                    cudaStream_t st, bool ppm)
{
    const bool m = psi || alp;
    if (ppm)
        return m ? stencil_launch<true, T, true>(g, prim, bf, psi, alp, F, fe, Eh, nsm, st)
                 : stencil_launch<false, T, true>(g, prim, bf, psi, alp, F, fe, Eh, nsm, st);
    return m ? stencil_launch<true, T, false>(g, prim, bf, psi, alp, F, fe, Eh, nsm, st)
             : stencil_launch<false, T, false>(g, prim, bf, psi, alp, F, fe, Eh, nsm, st);
}

cudaError_t launch_stencil32(const Dims& g, const PrimIn<float>& prim, CP3 bf, const double* psi, const double* alp,
                             const FluxOut<float>* F, double* const (*fe)[3], double* const* Eh, int nsm,
                             cudaStream_t st, bool ppm)
{
    return stencil_dispatch<float>(g, prim, bf, psi, alp, F, fe, Eh, nsm, st, ppm);
}

cudaError_t launch_stencil64(const Dims& g, CP8 prim, CP3 bf, const double* psi, const double* alp, const P8* F,
                             double* const (*fe)[3], double* const* Eh, int nsm, cudaStream_t st, bool ppm)
{
    PrimIn<double> p;
    FluxOut<double> fo[3];
    for (int v = 0; v < 8; v++) p.p[v] = prim.p[v];
    for (int d = 0; d < 3; d++)
        for (int v = 0; v < 8; v++) fo[d].p[v] = F[d].p[v];
    return stencil_dispatch<double>(g, p, bf, psi, alp, fo, fe, Eh, nsm, st, ppm);
}

cudaError_t launch_update(const Dims& g, const UpdateArgs& a, int nsm, cudaStream_t st)
{
    long long work = 1;
    for (int d = 0; d < 3; d++) work *= g.act[d] ? g.n[d] + 1 : 1;
    const int b = grid_for(work, 128, nsm);
    const bool m = a.psi || a.alp;
    if (a.f32 && b <= nsm * kUpdateSmall)
        launch_k(m ? k_update<true, true, true> : k_update<false, true, true>, b, 128, st, g, a);
    else if (a.f32) launch_k(m ? k_update<true, true> : k_update<false, true>, b, 128, st, g, a);
    else launch_k(m ? k_update<true, false> : k_update<false, false>, b, 128, st, g, a);
    return cudaGetLastError();
}

cudaError_t launch_curlA(const Dims& g, CP3 A, P3 bf, int nsm, cudaStream_t st)
{
    k_curlA<<<grid_for(g.ncell, 256, nsm), 256, 0, st>>>(g, A, bf);
    return cudaGetLastError();
}

cudaError_t launch_prim2con(const Dims& g, CP8 prim, CP3 bf, const double* psi, P8 q, int nsm, cudaStream_t st)
{
    k_prim2con<<<grid_for(g.ncell, 256, nsm), 256, 0, st>>>(g, prim, bf, psi, q);
    return cudaGetLastError();
}

cudaError_t launch_prim_to32(const Dims& g, CP8 prim, CP3 bf, F11 p32, int nsm, cudaStream_t st)
{
    k_prim_to32<<<grid_for(g.ncell, 256, nsm), 256, 0, st>>>(g, prim, bf, p32);
    return cudaGetLastError();
}

cudaError_t launch_dt(const Dims& g, const double* psi, const double* alp, double* part, int nblk, double* out,
                      cudaStream_t st)
{
    k_dt<<<nblk, 256, 0, st>>>(g, psi, alp, part);
    k_fold<<<1, 256, 0, st>>>(part, nblk, 1, nullptr, 1u, out);
    return cudaGetLastError();
}

cudaError_t launch_diag(const Dims& g, CP3 bf, CP8 q, double dV, double* part, int nblk, double* out,
                        cudaStream_t st)
{
    k_diag<<<nblk, 256, 0, st>>>(g, bf, q, dV, part);
    k_fold<<<1, 256, 0, st>>>(part, nblk, 11, nullptr, 1u << 2, out);
    return cudaGetLastError();
}

cudaError_t launch_curlA_cc(const Dims& g, CP3 A, P3 qB, int nsm, cudaStream_t st)
{
    k_curlA_cc<<<grid_for((long long)g.n[0] * g.n[1] * g.n[2], 256, nsm), 256, 0, st>>>(g, A, qB);
    return cudaGetLastError();
}

cudaError_t launch_prim2con_cc(const Dims& g, CP8 prim, CP3 qB, const double* psi, const double* phi, double* qphi,
                               P8 q, int nsm, cudaStream_t st)
{
    k_prim2con_cc<<<grid_for(g.ncell, 256, nsm), 256, 0, st>>>(g, prim, qB, psi, phi, qphi, q);
    return cudaGetLastError();
}

cudaError_t launch_diag_cc(const Dims& g, CP3 qB, CP8 q, double dV, double* part, int nblk, double* out,
                           cudaStream_t st)
{
    k_diag_cc<<<nblk, 256, 0, st>>>(g, qB, q, dV, part);
    k_fold<<<1, 256, 0, st>>>(part, nblk, 11, nullptr, 1u << 2, out);
    return cudaGetLastError();
}

GRMHD_OOB_READER(oob_kernels)

}  // namespace grmhd
