// Elliptic divergence cleaning (arXiv 2110.03732 Sec. 3.3) by geometric multigrid,
// sm_103a, FP64: solve lap(Phi) = div q_B and set q_B <- q_B - grad(Phi).
//
// Operators (Cartesian reference metric, so flat):
//   staggered fields (CT): div on cells from face differences, grad on faces from the
//     two adjacent cells; lap = div(grad) is the compact (2 ndim + 1)-point stencil and
//     the cleaned field is divergence-free to the solver's accuracy;
//   cell-centred fields (GLM): div and grad by central differences with the same
//     compact lap (an approximate projection).
//   Periodic directions wrap; in the others Phi has zero normal gradient (no flux
//   through the boundary face, which is not corrected).  The right-hand side is made
//   mean-free (the constants are the null space).
//
// Multigrid: cell-centred levels, each halving every active extent while all of them
// are even and at least 4.  V(2,2) cycles: red-black Gauss-Seidel smoothing (valid,
// hence deterministic, because every level but the coarsest has even extents), the
// residual of the 2^ndim children averaged to the coarse cell, tensor-product linear
// interpolation (weights 3/4, 1/4) back.  The coarsest level (at most 4096 cells) is
// solved by conjugate gradients in one thread block with fixed-order reductions and
// a bounded iteration count.  Every launch is deterministic; the cycle count is fixed
// by the caller, so a cleaning is launches only (no host synchronisation).
#include <cuda_runtime.h>

#include "elliptic.h"
#include "grmhd_device.cuh"
#include "launch.cuh"

namespace grmhd {

namespace {

// cell (i, j, k) of a level, x fastest; returns the neighbour's index along d (side s =
// +-1), or -1 past a non-periodic boundary
__device__ __forceinline__ long long mg_nb(const MgLevel& L, const int* bc, int i, int j, int k, int d, int s)
{
    int c[3] = {i, j, k};
    c[d] += s;
    if (c[d] < 0 || c[d] >= L.n[d]) {
        if (bc[d] != BC_PERIODIC) return -1;
        c[d] += c[d] < 0 ? L.n[d] : -L.n[d];
    }
    return c[0] + (long long)L.n[0] * (c[1] + (long long)L.n[1] * c[2]);
}

struct MgArgs {
    int bc[3];
    int act[3];
};

// cell (i, j, k) of level item t (levels hold fewer than 2^31 cells: mg_plan); a division
// by a run-time value would issue its conversions on the FP64 pipe
__device__ __forceinline__ void mg_coords(const MgLevel& L, long long t, int& i, int& j, int& k)
{
    int c[3];
    box_coords(t, L.f0, L.f1, c);
    i = c[0];
    j = c[1];
    k = c[2];
}

// (L Phi)_c split as sum_nb Phi_nb / h^2 - diag Phi_c; returns the neighbour sum, the
// diagonal and the number of neighbours missing past non-periodic boundaries (0: the
// full stencil, whose diagonal is the level's dfull)
__device__ __forceinline__ void mg_stencil(const MgLevel& L, const MgArgs& m, const double* __restrict__ phi, int i,
                                           int j, int k, double& nbsum, double& diag, int& miss)
{
    nbsum = 0.0;
    miss = 0;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        if (!m.act[d]) continue;
        const long long lo = mg_nb(L, m.bc, i, j, k, d, -1), hi = mg_nb(L, m.bc, i, j, k, d, 1);
        double s2;
        if (lo >= 0 && hi >= 0) {
            s2 = phi[lo] + phi[hi];
        } else {
            s2 = lo >= 0 ? phi[lo] : (hi >= 0 ? phi[hi] : 0.0);
            miss += (lo < 0) + (hi < 0);
        }
        nbsum += s2 * L.ih2[d];
    }
    diag = L.dfull;
    if (miss) {
        diag = 0.0;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            if (!m.act[d]) continue;
            if (mg_nb(L, m.bc, i, j, k, d, -1) >= 0) diag += L.ih2[d];
            if (mg_nb(L, m.bc, i, j, k, d, 1) >= 0) diag += L.ih2[d];
        }
    }
}

// cells of colour `color` ((i + j + k) & 1) of a level, enumerated x fastest: item t
// is the u-th such cell of row (j, k), u = t mod ceil(n_x / 2)
__device__ __forceinline__ long long mg_half_items(const MgLevel& L)
{
    return (long long)((L.n[0] + 1) >> 1) * L.n[1] * L.n[2];
}

// red-black Gauss-Seidel update of item t of colour `color`.  The full stencil's
// diagonal reciprocal is the level's; a boundary cell (fewer neighbours) divides.
__device__ __forceinline__ void mg_smooth_cell(const MgLevel& L, const MgArgs& m, int color, long long t)
{
    int x[3];
    box_coords(t, L.fh, L.f1, x);
    const int j = x[1], k = x[2];
    const int i = 2 * x[0] + ((color + j + k) & 1);
    if (i >= L.n[0]) return;
    const int c = i + L.n[0] * (j + L.n[1] * k);
    double nbsum, diag;
    int miss;
    mg_stencil(L, m, L.phi, i, j, k, nbsum, diag, miss);
    if (!miss) L.phi[c] = (nbsum - L.rhs[c]) * L.idiag;
    else if (diag > 0.0) L.phi[c] = (nbsum - L.rhs[c]) / diag;
}

__global__ void __launch_bounds__(256) k_mg_smooth(MgLevel L, MgArgs m, int color)
{
    grid_dep_sync();
    const long long items = mg_half_items(L);
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < items;
         t += (long long)gridDim.x * blockDim.x)
        mg_smooth_cell(L, m, color, t);
}

// coarse rhs of cell t = mean of its children's residuals rhs - L Phi; coarse Phi = 0
__device__ __forceinline__ void mg_restrict_cell(const MgLevel& F, const MgLevel& C, const MgArgs& m, long long t)
{
    {
        int I, J, K;
        mg_coords(C, t, I, J, K);
        double sum = 0.0;
        for (int dk = 0; dk <= m.act[2]; dk++)
            for (int dj = 0; dj <= m.act[1]; dj++)
                for (int di = 0; di <= m.act[0]; di++) {
                    const int i = 2 * I * m.act[0] + di, j = 2 * J * m.act[1] + dj, k = 2 * K * m.act[2] + dk;
                    const long long f = i + (long long)F.n[0] * (j + (long long)F.n[1] * k);
                    double nbsum, diag;
                    int miss;
                    mg_stencil(F, m, F.phi, i, j, k, nbsum, diag, miss);
                    sum += F.rhs[f] - (nbsum - diag * F.phi[f]);
                }
        // 1 / (number of children), a power of two
        C.rhs[t] = sum * ((m.act[0] ? 0.5 : 1.0) * (m.act[1] ? 0.5 : 1.0) * (m.act[2] ? 0.5 : 1.0));
        C.phi[t] = 0.0;
    }
}

__global__ void __launch_bounds__(256) k_mg_restrict(MgLevel F, MgLevel C, MgArgs m)
{
    grid_dep_sync();
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < C.cells;
         t += (long long)gridDim.x * blockDim.x)
        mg_restrict_cell(F, C, m, t);
}

// Phi_fine += linear interpolation of the coarse correction: along each active
// direction the child takes 3/4 of its parent and 1/4 of the parent's neighbour on its
// side (the parent itself past a non-periodic boundary)
__device__ __forceinline__ void mg_prolong_cell(const MgLevel& F, const MgLevel& C, const MgArgs& m, long long t)
{
    {
        int c[3];
        mg_coords(F, t, c[0], c[1], c[2]);
        int P[3], S[3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            P[d] = m.act[d] ? c[d] >> 1 : c[d];
            S[d] = m.act[d] ? ((c[d] & 1) ? 1 : -1) : 0;
        }
        double v = 0.0;
        for (int ok = 0; ok <= m.act[2]; ok++)
            for (int oj = 0; oj <= m.act[1]; oj++)
                for (int oi = 0; oi <= m.act[0]; oi++) {
                    const int off[3] = {oi, oj, ok};
                    int q[3];
                    double w = 1.0;
                    for (int d = 0; d < 3; d++) {
                        if (!m.act[d]) { q[d] = P[d]; continue; }
                        q[d] = P[d] + off[d] * S[d];
                        w *= off[d] ? 0.25 : 0.75;
                        if (q[d] < 0 || q[d] >= C.n[d]) {
                            if (m.bc[d] == BC_PERIODIC) q[d] += q[d] < 0 ? C.n[d] : -C.n[d];
                            else q[d] = P[d];
                        }
                    }
                    v += w * C.phi[q[0] + (long long)C.n[0] * (q[1] + (long long)C.n[1] * q[2])];
                }
        F.phi[t] += v;
    }
}

__global__ void __launch_bounds__(256) k_mg_prolong(MgLevel F, MgLevel C, MgArgs m)
{
    grid_dep_sync();
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < F.cells;
         t += (long long)gridDim.x * blockDim.x)
        mg_prolong_cell(F, C, m, t);
}

// fixed-order block sum (blockDim.x a multiple of 32, at most 1024)
__device__ __forceinline__ double mg_block_sum(double v, double* sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        v = l < (int)(blockDim.x >> 5) ? sh[l] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (l == 0) sh[32] = v;
    }
    __syncthreads();
    return sh[32];
}

// the block sum where one warp holds every value: five shuffles.  Shuffles order no memory, so a
// warp barrier stands before them: what the lanes wrote before the sum is read after it by
// others (the search direction), as with the barriers of the block sum.
template <bool W>
__device__ __forceinline__ double mg_sum(double v, double* sh)
{
    if (!W) return mg_block_sum(v, sh);
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <bool W>
__device__ __forceinline__ void mg_sync()
{
    if (W) __syncwarp();
    else __syncthreads();
}

// coarsest level: conjugate gradients on -lap (symmetric positive semi-definite) with
// a mean-free right-hand side, in one block.  r, p and q are scratch vectors of the
// level's size; iterations end at ||r|| <= 1e-15 ||b|| or after max_it.
//
// W: by the first warp alone (the callers' other warps wait), for a level of so few cells
// that the block barriers of the sums would cost more than the arithmetic. 
template <bool W>
__device__ __forceinline__ void mg_cg_run(const MgLevel& L, const MgArgs& m, double* __restrict__ res,
                                          double* __restrict__ p, double* __restrict__ q, int max_it, double* sh)
{
    const int n = (int)L.cells, nt = W ? 32 : (int)blockDim.x;
    // b = -(rhs - mean rhs); x = 0, r = b, p = r
    double s = 0.0;
    for (int t = threadIdx.x; t < n; t += nt) s += L.rhs[t];
    const double mean = mg_sum<W>(s, sh) / (double)n;
    double rr = 0.0;
    for (int t = threadIdx.x; t < n; t += nt) {
        const double b = -(L.rhs[t] - mean);
        res[t] = b;
        p[t] = b;
        L.phi[t] = 0.0;
        rr += b * b;
    }
    rr = mg_sum<W>(rr, sh);
    const double stop = 1e-30 * rr;
    for (int it = 0; it < max_it && rr > stop && rr > 0.0; it++) {
        // q = -lap p
        double pq = 0.0;
        for (int t = threadIdx.x; t < n; t += nt) {
            int i, j, k;
            mg_coords(L, t, i, j, k);
            double nbsum, diag;
            int miss;
            mg_stencil(L, m, p, i, j, k, nbsum, diag, miss);
            const double v = diag * p[t] - nbsum;
            q[t] = v;
            pq += p[t] * v;
        }
        pq = mg_sum<W>(pq, sh);
        if (!(pq > 0.0)) break;
        const double alpha = rr / pq;
        double rn = 0.0;
        for (int t = threadIdx.x; t < n; t += nt) {
            L.phi[t] += alpha * p[t];
            const double r = res[t] - alpha * q[t];
            res[t] = r;
            rn += r * r;
        }
        rn = mg_sum<W>(rn, sh);
        const double beta = rn / rr;
        rr = rn;
        for (int t = threadIdx.x; t < n; t += nt) p[t] = res[t] + beta * p[t];
        mg_sync<W>();
    }
    mg_sync<W>();
}

__device__ __forceinline__ void mg_cg_block(const MgLevel& L, const MgArgs& m, double* __restrict__ res,
                                            double* __restrict__ p, double* __restrict__ q, int max_it, double* sh)
{
    if (L.cells <= 64) {
        if (threadIdx.x < 32) mg_cg_run<true>(L, m, res, p, q, max_it, sh);
        __syncthreads();
    } else {
        mg_cg_run<false>(L, m, res, p, q, max_it, sh);
    }
}

// the levels first..nlev-1 (each at most kMgBlockCells cells) of one V-cycle in a
// single block: down-leg smoothing and restriction, conjugate gradients on the
// coarsest, up-leg interpolation and smoothing -- the same updates in the same order
// as the one-launch-per-step form, with block barriers in place of launches.  With
// smem set the block moves these levels and the CG vectors into dynamic shared memory
// (level `first` in from its global arrays at the start, its Phi back at the end).
struct MgTail {
    MgLevel lev[kMgMaxLevels];
    long long soff[kMgMaxLevels];   // with smem: offset (doubles) of each tail level's
                                    // Phi (its rhs follows) in the shared block
    long long scg;                  // with smem: offset of the CG vectors r, p, q
    int first, nlev;
    int smem;
};

// level l of the tail with its arrays where the block keeps them (a register copy: the
// kernel's parameter block itself is never written, which would move it to local memory)
__device__ __forceinline__ MgLevel tail_level(const MgTail& T, int l, double* sm)
{
    MgLevel L = T.lev[l];
    if (T.smem) {
        L.phi = sm + T.soff[l];
        L.rhs = L.phi + L.cells;
    }
    return L;
}

__global__ void __launch_bounds__(1024) k_mg_tail(MgTail T, MgArgs m, double* __restrict__ res,
                                                   double* __restrict__ p, double* __restrict__ q, int max_it)
{
    grid_dep_sync();
    extern __shared__ double tail_sm[];
    __shared__ double sh[kMgSums];
    if (T.smem) {
        const MgLevel G = T.lev[T.first];
        const MgLevel L = tail_level(T, T.first, tail_sm);
        for (long long t = threadIdx.x; t < L.cells; t += blockDim.x) {
            L.phi[t] = G.phi[t];
            L.rhs[t] = G.rhs[t];
        }
        const long long nc = T.lev[T.nlev - 1].cells;
        res = tail_sm + T.scg;
        p = res + nc;
        q = p + nc;
        __syncthreads();
    }
    for (int l = T.first; l + 1 < T.nlev; l++) {
        const MgLevel L = tail_level(T, l, tail_sm), C = tail_level(T, l + 1, tail_sm);
        const long long items = mg_half_items(L);
        for (int s = 0; s < 2; s++)
            for (int color = 0; color < 2; color++) {
                for (long long t = threadIdx.x; t < items; t += blockDim.x) mg_smooth_cell(L, m, color, t);
                __syncthreads();
            }
        for (long long t = threadIdx.x; t < C.cells; t += blockDim.x) mg_restrict_cell(L, C, m, t);
        __syncthreads();
    }
    mg_cg_block(tail_level(T, T.nlev - 1, tail_sm), m, res, p, q, max_it, sh);
    for (int l = T.nlev - 2; l >= T.first; l--) {
        const MgLevel L = tail_level(T, l, tail_sm), C = tail_level(T, l + 1, tail_sm);
        for (long long t = threadIdx.x; t < L.cells; t += blockDim.x) mg_prolong_cell(L, C, m, t);
        __syncthreads();
        const long long items = mg_half_items(L);
        for (int s = 0; s < 2; s++)
            for (int color = 0; color < 2; color++) {
                for (long long t = threadIdx.x; t < items; t += blockDim.x) mg_smooth_cell(L, m, color, t);
                __syncthreads();
            }
    }
    if (T.smem) {
        const MgLevel G = T.lev[T.first];
        const MgLevel L = tail_level(T, T.first, tail_sm);
        for (long long t = threadIdx.x; t < L.cells; t += blockDim.x) G.phi[t] = L.phi[t];
    }
}

// ---------------------------------------------------------------------------
// 2-D levels: the four half sweeps of a leg and its transfer in one launch
// ---------------------------------------------------------------------------

// A block owns a T x T tile and holds it with a halo of H cells in shared memory.  Half sweep
// s updates the cells up to H - 1 - s from the tile (those of its colour), so that each
// needs only cells the half sweep before has updated: every cell gets the value the
// grid-wide half sweeps give it (to rounding), the halo's being computed by each block that
// needs them.  The legs write to the level's other Phi array, since a block's halo is
// another block's tile.  A leg took five launches of 4-9 us, each a few hundred cycles of
// work; the redundant halo cells cost less than those.
template <int T, int H>
struct MgTile {
    static constexpr int R = T + 2 * H;
    double phi[R][R + 1], rs[R][R + 1];   // Phi and rhs / diagonal of the full stencil
};

// level coordinate of region coordinate r of a tile at o: wrapped, or -1 outside a
// non-periodic extent (o - H + 2n >= 0: fused levels have n >= 4)
__device__ __forceinline__ int mg_wrap(int x, int n, const FastDiv& f, bool periodic)
{
    if (x >= 0 && x < n) return x;
    if (!periodic) return -1;
    const unsigned u = (unsigned)(x + 2 * n);
    return (int)(u - fdiv(u, f) * (unsigned)n);
}

// Phi of the region cell (rx, ry) by one Gauss-Seidel update; x, y its level coordinates.
// A cell beside a non-periodic boundary has fewer neighbours and divides.
template <int T, int H>
__device__ __forceinline__ double mg_tile_update(const MgLevel& L, const MgArgs& m, const MgTile<T, H>& S, int rx,
                                                 int ry, int x, int y)
{
    const bool bx = m.bc[0] != BC_PERIODIC && (x == 0 || x == L.n[0] - 1);
    const bool by = m.bc[1] != BC_PERIODIC && (y == 0 || y == L.n[1] - 1);
    const double l = S.phi[ry][rx - 1], r = S.phi[ry][rx + 1], d = S.phi[ry - 1][rx], u = S.phi[ry + 1][rx];
    if (!bx && !by) return fma(l + r, L.cx[0], fma(d + u, L.cx[1], -S.rs[ry][rx]));
    double nb = 0.0, diag = 0.0;
    if (!(bx && x == 0)) { nb += l * L.ih2[0]; diag += L.ih2[0]; }
    if (!(bx && x == L.n[0] - 1)) { nb += r * L.ih2[0]; diag += L.ih2[0]; }
    if (!(by && y == 0)) { nb += d * L.ih2[1]; diag += L.ih2[1]; }
    if (!(by && y == L.n[1] - 1)) { nb += u * L.ih2[1]; diag += L.ih2[1]; }
    return diag > 0.0 ? (nb - S.rs[ry][rx] * L.dfull) / diag : S.phi[ry][rx];
}

template <int T, int H>
__device__ __forceinline__ void mg_tile_sweeps(const MgLevel& L, const MgArgs& m, MgTile<T, H>& S, int ox, int oy)
{
    const bool px = m.bc[0] == BC_PERIODIC, py = m.bc[1] == BC_PERIODIC;
#pragma unroll
    for (int s = 0; s < 4; s++) {
        constexpr int e0 = H - 1;
        const int e = e0 - s, w = T + 2 * e, hw = w / 2;   // T + 2e is even
        __syncthreads();
        for (int t = threadIdx.x; t < w * hw; t += blockDim.x) {
            const int row = t / hw, ry = H - e + row;
            const int y = oy + ry - H;
            // colour (x + y) & 1 of the unwrapped coordinates: extents are even
            const int rx0 = H - e, x0 = ox + rx0 - H;
            const int rx = rx0 + 2 * (t - row * hw) + ((x0 + y + s) & 1);
            const int gx = mg_wrap(ox + rx - H, L.n[0], L.f0, px), gy = mg_wrap(y, L.n[1], L.f1, py);
            if (gx < 0 || gy < 0) continue;
            S.phi[ry][rx] = mg_tile_update<T, H>(L, m, S, rx, ry, gx, gy);
        }
    }
    __syncthreads();
}

// down leg: four half sweeps from L.phi (zero: from 0), Phi to L.alt, the residual averaged
// to the coarse right-hand side, and the coarse Phi set to zero
template <int T>
__global__ void __launch_bounds__(256) k_mg_down2(MgLevel L, MgLevel C, MgArgs m, int zero)
{
    constexpr int H = 5;
    __shared__ MgTile<T, H> S;
    grid_dep_sync();
    const int ox = blockIdx.x * T, oy = blockIdx.y * T;
    constexpr int R = MgTile<T, H>::R;
    for (int t = threadIdx.x; t < R * R; t += blockDim.x) {
        const int ry = t / R, rx = t - ry * R;
        const int gx = mg_wrap(ox + rx - H, L.n[0], L.f0, m.bc[0] == BC_PERIODIC);
        const int gy = mg_wrap(oy + ry - H, L.n[1], L.f1, m.bc[1] == BC_PERIODIC);
        const bool in = gx >= 0 && gy >= 0;
        const long long c = in ? gx + (long long)L.n[0] * gy : 0;
        S.phi[ry][rx] = in && !zero ? L.phi[c] : 0.0;
        S.rs[ry][rx] = in ? L.rhs[c] * L.idiag : 0.0;
    }
    mg_tile_sweeps<T, H>(L, m, S, ox, oy);
    for (int t = threadIdx.x; t < T * T; t += blockDim.x) {
        const int ty = t / T, tx = t - ty * T;
        if (ox + tx < L.n[0] && oy + ty < L.n[1])
            L.alt[ox + tx + (long long)L.n[0] * (oy + ty)] = S.phi[ty + H][tx + H];
    }
    for (int t = threadIdx.x; t < T * T / 4; t += blockDim.x) {
        const int cy = t / (T / 2), cx = t - cy * (T / 2);
        const int X = ox / 2 + cx, Y = oy / 2 + cy;
        if (X >= C.n[0] || Y >= C.n[1]) continue;
        double sum = 0.0;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int rx = 2 * cx + (k & 1) + H, ry = 2 * cy + (k >> 1) + H;
            const int x = ox + rx - H, y = oy + ry - H;
            const bool edge = (m.bc[0] != BC_PERIODIC && (x == 0 || x == L.n[0] - 1)) ||
                              (m.bc[1] != BC_PERIODIC && (y == 0 || y == L.n[1] - 1));
            const double f = S.phi[ry][rx];
            if (!edge) {
                // residual / dfull = rs - (neighbour sum) idiag + Phi
                sum += (S.rs[ry][rx] + f) - fma(S.phi[ry][rx - 1] + S.phi[ry][rx + 1], L.cx[0],
                                                (S.phi[ry - 1][rx] + S.phi[ry + 1][rx]) * L.cx[1]);
            } else {
                double r = S.rs[ry][rx] * L.dfull;
                if (m.bc[0] == BC_PERIODIC || x > 0) r -= (S.phi[ry][rx - 1] - f) * L.ih2[0];
                if (m.bc[0] == BC_PERIODIC || x < L.n[0] - 1) r -= (S.phi[ry][rx + 1] - f) * L.ih2[0];
                if (m.bc[1] == BC_PERIODIC || y > 0) r -= (S.phi[ry - 1][rx] - f) * L.ih2[1];
                if (m.bc[1] == BC_PERIODIC || y < L.n[1] - 1) r -= (S.phi[ry + 1][rx] - f) * L.ih2[1];
                sum += r * L.idiag;
            }
        }
        const long long c = X + (long long)C.n[0] * Y;
        C.rhs[c] = sum * (0.25 * L.dfull);
        C.phi[c] = 0.0;
    }
}

// up leg: the coarse correction interpolated onto L.alt (as mg_prolong_cell), then four half
// sweeps; Phi to L.phi
template <int T>
__global__ void __launch_bounds__(256) k_mg_up2(MgLevel L, MgLevel C, MgArgs m)
{
    constexpr int H = 4;
    __shared__ MgTile<T, H> S;
    grid_dep_sync();
    const int ox = blockIdx.x * T, oy = blockIdx.y * T;
    constexpr int R = MgTile<T, H>::R;
    const bool px = m.bc[0] == BC_PERIODIC, py = m.bc[1] == BC_PERIODIC;
    for (int t = threadIdx.x; t < R * R; t += blockDim.x) {
        const int ry = t / R, rx = t - ry * R;
        const int gx = mg_wrap(ox + rx - H, L.n[0], L.f0, px), gy = mg_wrap(oy + ry - H, L.n[1], L.f1, py);
        double v = 0.0, rs = 0.0;
        if (gx >= 0 && gy >= 0) {
            const long long c = gx + (long long)L.n[0] * gy;
            rs = L.rhs[c] * L.idiag;
            const int X = gx >> 1, Y = gy >> 1;
            int X1 = X + ((gx & 1) ? 1 : -1), Y1 = Y + ((gy & 1) ? 1 : -1);
            if (X1 < 0 || X1 >= C.n[0]) X1 = px ? (X1 < 0 ? X1 + C.n[0] : X1 - C.n[0]) : X;
            if (Y1 < 0 || Y1 >= C.n[1]) Y1 = py ? (Y1 < 0 ? Y1 + C.n[1] : Y1 - C.n[1]) : Y;
            const long long r0 = (long long)C.n[0] * Y, r1 = (long long)C.n[0] * Y1;
            const double a = fma(0.25, C.phi[X1 + r0], 0.75 * C.phi[X + r0]);
            const double b = fma(0.25, C.phi[X1 + r1], 0.75 * C.phi[X + r1]);
            v = fma(0.25, b, fma(0.75, a, L.alt[c]));
        }
        S.phi[ry][rx] = v;
        S.rs[ry][rx] = rs;
    }
    mg_tile_sweeps<T, H>(L, m, S, ox, oy);
    for (int t = threadIdx.x; t < T * T; t += blockDim.x) {
        const int ty = t / T, tx = t - ty * T;
        if (ox + tx < L.n[0] && oy + ty < L.n[1])
            L.phi[ox + tx + (long long)L.n[0] * (oy + ty)] = S.phi[ty + H][tx + H];
    }
}

// fine right-hand side: div q_B on the interior cells (faces or central), and block
// partial sums for its mean
__global__ void __launch_bounds__(256) k_mg_div(Dims g, CP3 bq, int cc, MgLevel L, MgArgs m, double* __restrict__ part)
{
    grid_dep_sync();
    __shared__ double sh[kMgSums];
    double s = 0.0;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < L.cells;
         t += (long long)gridDim.x * blockDim.x) {
        int c[3];
        mg_coords(L, t, c[0], c[1], c[2]);
        int p[3] = {c[0] + g.ng[0], c[1] + g.ng[1], c[2] + g.ng[2]};
        const long long o = lin(g, p[0], p[1], p[2]);
        double dv = 0.0;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            if (!g.act[d]) continue;
            if (cc) {
                // central difference; past a non-periodic boundary the cell itself (zero
                // gradient, whatever the boundary kind)
                const long long hi = mg_nb(L, m.bc, c[0], c[1], c[2], d, 1);
                const long long lo = mg_nb(L, m.bc, c[0], c[1], c[2], d, -1);
                int ch[3] = {c[0], c[1], c[2]}, cl[3] = {c[0], c[1], c[2]};
                if (hi >= 0) ch[d] = (c[d] + 1) % L.n[d];
                if (lo >= 0) cl[d] = (c[d] - 1 + L.n[d]) % L.n[d];
                const double vh = bq.p[d][lin(g, ch[0] + g.ng[0], ch[1] + g.ng[1], ch[2] + g.ng[2])];
                const double vl = bq.p[d][lin(g, cl[0] + g.ng[0], cl[1] + g.ng[1], cl[2] + g.ng[2])];
                dv += (vh - vl) * (0.5 * g.idx[d]);
            } else {
                int up[3] = {p[0], p[1], p[2]};
                up[d] += 1;
                dv += (bq.p[d][face_at(g, d, up)] - bq.p[d][o]) * g.idx[d];
            }
        }
        L.rhs[t] = dv;
        L.phi[t] = 0.0;
        s += dv;
    }
    s = mg_block_sum(s, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// mean of the partial sums (one block), subtracted from the fine right-hand side
__global__ void __launch_bounds__(256) k_mg_mean(const double* __restrict__ part, int nb, double* __restrict__ mean,
                                                 long long cells)
{
    grid_dep_sync();
    __shared__ double sh[kMgSums];
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) s += part[b];
    s = mg_block_sum(s, sh);
    if (threadIdx.x == 0) *mean = s / (double)cells;
}

__global__ void __launch_bounds__(256) k_mg_sub_mean(MgLevel L, const double* __restrict__ mean)
{
    grid_dep_sync();
    const double mu = *mean;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < L.cells;
         t += (long long)gridDim.x * blockDim.x)
        L.rhs[t] -= mu;
}

// q_B -= grad Phi: staggered (lower face of each interior cell; the lower boundary face
// of a non-periodic direction is kept) or central (cell-centred)
__global__ void __launch_bounds__(256) k_mg_correct(Dims g, P3 bq, int cc, MgLevel L, MgArgs m)
{
    grid_dep_sync();
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < L.cells;
         t += (long long)gridDim.x * blockDim.x) {
        int c[3];
        mg_coords(L, t, c[0], c[1], c[2]);
        const long long o = lin(g, c[0] + g.ng[0], c[1] + g.ng[1], c[2] + g.ng[2]);
#pragma unroll
        for (int d = 0; d < 3; d++) {
            if (!g.act[d]) continue;
            const long long lo = mg_nb(L, m.bc, c[0], c[1], c[2], d, -1);
            if (cc) {
                const long long hi = mg_nb(L, m.bc, c[0], c[1], c[2], d, 1);
                const double pl = lo < 0 ? L.phi[t] : L.phi[lo];
                const double ph = hi < 0 ? L.phi[t] : L.phi[hi];
                bq.p[d][o] -= (ph - pl) * (0.5 * g.idx[d]);
            } else if (lo >= 0) {
                bq.p[d][o] -= (L.phi[t] - L.phi[lo]) * g.idx[d];
            }
        }
    }
}

// items of one colour of a level (mg_half_items on the host)
long long half_items(const MgLevel& L)
{
    return (long long)((L.n[0] + 1) / 2) * L.n[1] * L.n[2];
}

int mg_grid(long long work, int nsm)
{
    long long b = (work + 255) / 256;
    const long long cap = (long long)nsm * 8;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

}  // namespace

int mg_plan(const Dims& g, MgPlan* plan)
{
    MgPlan p;
    p.nlev = 0;
    int n[3] = {g.n[0], g.n[1], g.n[2]};
    long long total = 0;
    for (;;) {
        if (p.nlev >= kMgMaxLevels) return -1;
        MgLevel& L = p.lev[p.nlev];
        long long cells = 1;
        for (int d = 0; d < 3; d++) {
            L.n[d] = n[d];
            const double h = g.act[d] ? (1.0 / g.idx[d]) * (double)(g.n[d] / n[d]) : 1.0;
            L.ih2[d] = g.act[d] ? 1.0 / (h * h) : 0.0;
            cells *= n[d];
        }
        // the device's summation order: per active direction, its two neighbours
        L.dfull = 0.0;
        for (int d = 0; d < 3; d++)
            if (g.act[d]) {
                L.dfull += L.ih2[d];
                L.dfull += L.ih2[d];
            }
        L.idiag = L.dfull > 0.0 ? 1.0 / L.dfull : 0.0;
        for (int d = 0; d < 3; d++) L.cx[d] = L.ih2[d] * L.idiag;
        L.f0 = make_fastdiv((unsigned)n[0]);
        L.f1 = make_fastdiv((unsigned)n[1]);
        L.fh = make_fastdiv((unsigned)((n[0] + 1) / 2));
        if (cells >= (1LL << 31)) return -3;
        L.cells = cells;
        L.offset = total;
        total += cells;
        p.nlev++;
        bool can = true;
        for (int d = 0; d < 3; d++)
            if (g.act[d] && (n[d] % 2 != 0 || n[d] < 4)) can = false;
        if (!can) break;
        for (int d = 0; d < 3; d++)
            if (g.act[d]) n[d] /= 2;
    }
    if (p.lev[p.nlev - 1].cells > kMgMaxCoarse) return -2;
    p.total = total;
    *plan = p;
    return 0;
}

size_t mg_scratch_bytes(const MgPlan& p)
{
    // phi and rhs of every level; CG vectors r, p, q of the coarsest; partial sums; mean
    const size_t coarse = (size_t)p.lev[p.nlev - 1].cells;
    return sizeof(double) * (2 * (size_t)p.total + 3 * coarse + kMgParts + 1);
}

cudaError_t mg_clean(const Dims& g, const MgPlan& plan0, double* scratch, double* alt0, double* alt1,
                     double* const* bq, bool cc, int cycles, int nsm, cudaStream_t st, long long* launches)
{
    // launches, up to the first that is refused: what comes after one, the field's correction
    // above all, would work on a level that was not computed
    long long nl = 0;
    cudaError_t err = cudaSuccess;
    auto go = [&](auto* k, dim3 grid, int block, size_t smem, auto&&... args) {
        if (err != cudaSuccess) return;
        nl++;
        err = launch_dyn(k, grid, block, smem, st, args...);
    };
    MgPlan plan = plan0;
    const long long T = plan.total;
    const long long nc = plan.lev[plan.nlev - 1].cells;
    for (int l = 0; l < plan.nlev; l++) {
        MgLevel& L = plan.lev[l];
        L.phi = scratch + L.offset;
        L.rhs = scratch + T + L.offset;
        L.alt = l == 0 ? alt0 : alt1 + (L.offset - plan.lev[0].cells);
    }
    double* cg_r = scratch + 2 * T;
    double* cg_p = cg_r + nc;
    double* cg_q = cg_p + nc;
    double* part = cg_q + nc;
    double* mean = part + kMgParts;
    MgArgs m;
    for (int d = 0; d < 3; d++) {
        m.bc[d] = g.bc[d];
        m.act[d] = g.act[d];
    }
    const MgLevel& F = plan.lev[0];
    CP3 cq;
    P3 pq;
    for (int d = 0; d < 3; d++) {
        cq.p[d] = bq[d];
        pq.p[d] = bq[d];
    }
    const int nb = (int)((F.cells + 255) / 256 < kMgParts ? (F.cells + 255) / 256 : kMgParts);
    go(k_mg_div, nb, 256, 0, g, cq, cc ? 1 : 0, F, m, part);
    go(k_mg_mean, 1, 256, 0, (const double*)part, nb, mean, F.cells);
    go(k_mg_sub_mean, mg_grid(F.cells, nsm), 256, 0, F, (const double*)mean);
    const int cg_it = (int)(2 * nc + 20);
    // levels of at most kMgBlockCells cells run inside one block (k_mg_tail)
    MgTail tail;
    for (int l = 0; l < plan.nlev; l++) tail.lev[l] = plan.lev[l];
    tail.nlev = plan.nlev;
    tail.first = plan.nlev - 1;
    while (tail.first > 0 && plan.lev[tail.first - 1].cells <= kMgBlockCells) tail.first--;
    long long soff = 0;
    for (int l = tail.first; l < plan.nlev; l++) {
        tail.soff[l] = soff;
        soff += 2 * plan.lev[l].cells;
    }
    tail.scg = soff;
    const size_t tail_bytes = sizeof(double) * (size_t)(soff + 3 * nc);
    tail.smem = tail_bytes <= kMgTailSmem ? 1 : 0;
    const size_t tail_dyn = tail.smem ? tail_bytes : 0;
    // 2-D levels: a leg per launch, in tiles of 32 cells a side where those fill the SMs, else 16
    const bool tiled = g.act[0] && g.act[1] && !g.act[2];
    auto tile_side = [&](const MgLevel& L) { return L.cells >= (long long)nsm * 1024 ? 32 : 16; };
    for (int cyc = 0; cyc < cycles; cyc++) {
        for (int l = 0; l < tail.first; l++) {
            const MgLevel& L = plan.lev[l];
            if (tiled) {
                const int T = tile_side(L);
                const dim3 gr((L.n[0] + T - 1) / T, (L.n[1] + T - 1) / T);
                go(T == 32 ? k_mg_down2<32> : k_mg_down2<16>, gr, 256, 0, L, plan.lev[l + 1], m,
                           (cyc == 0 || l > 0) ? 1 : 0);
                continue;
            }
            const int bs = mg_grid(half_items(L), nsm);
            for (int s = 0; s < 2; s++) {
                go(k_mg_smooth, bs, 256, 0, L, m, 0);
                go(k_mg_smooth, bs, 256, 0, L, m, 1);
            }
            go(k_mg_restrict, mg_grid(plan.lev[l + 1].cells, nsm), 256, 0, L, plan.lev[l + 1], m);
        }
        // the small levels and the coarsest solve (from zero); with a single level this
        // is the whole solve, and further cycles would repeat it
        go(k_mg_tail, 1, 1024, tail_dyn, tail, m, cg_r, cg_p, cg_q, cg_it);
        if (plan.nlev == 1) break;
        for (int l = tail.first - 1; l >= 0; l--) {
            const MgLevel& L = plan.lev[l];
            if (tiled) {
                const int T = tile_side(L);
                const dim3 gr((L.n[0] + T - 1) / T, (L.n[1] + T - 1) / T);
                go(T == 32 ? k_mg_up2<32> : k_mg_up2<16>, gr, 256, 0, L, plan.lev[l + 1], m);
                continue;
            }
            const int b = mg_grid(L.cells, nsm), bs = mg_grid(half_items(L), nsm);
            go(k_mg_prolong, b, 256, 0, L, plan.lev[l + 1], m);
            for (int s = 0; s < 2; s++) {
                go(k_mg_smooth, bs, 256, 0, L, m, 0);
                go(k_mg_smooth, bs, 256, 0, L, m, 1);
            }
        }
    }
    go(k_mg_correct, mg_grid(F.cells, nsm), 256, 0, g, pq, cc ? 1 : 0, F, m);
    if (launches) *launches += nl;
    const cudaError_t last = cudaGetLastError();   // (read in any case: it clears the error)
    return err != cudaSuccess ? err : last;
}

GRMHD_OOB_READER(oob_elliptic)

}  // namespace grmhd
