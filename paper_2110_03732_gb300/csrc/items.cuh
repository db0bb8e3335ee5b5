// Per-item bodies of the stage kernels (one cell, face or edge each), shared by
// the single-problem kernels (kernels.cu) and the batched multi-problem kernels
// (batch.cu), so that a problem advanced alone or inside a batch runs exactly the
// same arithmetic.  See kernels.cu for the paper passages each body follows.
#pragma once

#include "grmhd_device.cuh"
#include "kernels.h"

namespace grmhd {

// ---------------------------------------------------------------------------
// implicit step (Sec. 2.4): item t = interior cell t (x fastest)
// ---------------------------------------------------------------------------

// The outputs of a solved cell: primitives (FP64, and on the mixed path, F32, their FP32 copy
// from the caller's f32 = rho, u^1..3, p, E^1..3, q_B^1..3), the stiff rate R, the solved
// q_E and the history (uh: the FP32 orthonormal velocity, or NULL).  u and E orthonormal;
// qEs the stage base's q_E.
template <bool M, bool F32>
__device__ __forceinline__ void implicit_store(const ImpArgs& a, long long id, double rho, double pres,
                                               const double* u, const double* E, double ip2, double p4,
                                               const double* qEs, const float* f32, const float* uh)
{
    a.prim.p[0][id] = rho;
    a.prim.p[4][id] = pres;
    if (F32 && a.p32.p[0]) {
#pragma unroll
        for (int v = 0; v < 11; v++) a.p32.p[v][id] = f32[v];
    }
#pragma unroll
    for (int i = 0; i < 3; i++) {
        a.prim.p[1 + i][id] = M ? u[i] * ip2 : u[i];
        a.prim.p[5 + i][id] = M ? E[i] * ip2 : E[i];
        const double qEn = M ? p4 * E[i] : E[i];
        if (a.R.p[0]) a.R.p[i][id] = a.stiff ? (qEn - qEs[i]) * a.ia_dt : 0.0;
        if (a.qE_out.p[i]) a.qE_out.p[i][id] = qEn;
        if (a.hs[0] && uh) {
            a.hd[i][id] = uh[i] - a.hs[i][id];
            a.hs[i][id] = uh[i];
        }
    }
}

// the FP32 copies of a cell's primitives, converted on the integer pipe (a hardware
// conversion issues on the FP64 pipe)
template <bool M>
__device__ __forceinline__ void implicit_f32(double rho, double pres, const double* u, const double* E, double ip2,
                                             float* f32)
{
    f32[0] = d2f_int(rho);
    f32[4] = d2f_int(pres);
#pragma unroll
    for (int i = 0; i < 3; i++) {
        f32[1 + i] = d2f_int(M ? u[i] * ip2 : u[i]);
        f32[5 + i] = d2f_int(M ? E[i] * ip2 : E[i]);
    }
}

// The general solve of one cell (cells that implicit_item's direct path does not accept,
// and the dynamo form).
// refined: the direct path's double-word corrections have ended at (r0, r1, r2), and the
// solve goes on from there (from its start where that is not finite) without repeating them.
// CC: the magnetic field is cell-centred (a.bf holds cell q_B, GLM variant) instead of
// staggered on faces.  ACC: the mixed-precision path, whose double-word residual
// accepts the root (newton_refine_dw).  DYN: the dynamo form may apply (xi != 0)
template <bool M, bool CC, bool ACC, bool DYN>
__device__ __forceinline__ void implicit_solve(const Dims& g, const ImpArgs& a, long long t, bool refined, double r0,
                                               double r1, double r2)
{
    // flat metric: alpha = psi = 1 known at compile time
    const double* __restrict__ psi = M ? a.psi : nullptr;
    const double* __restrict__ alp = M ? a.alp : nullptr;
    const CP8& qb = a.qb;
    const CP3& bf = a.bf;
    const double* __restrict__ eta = a.eta;
    const double eta_u = a.eta_u, tol = a.tol, rho_atm = a.rho_atm, p_atm = a.p_atm;
    const int kmax = a.kmax;
    const P8& prim = a.prim;
    const P3& R = a.R;
    unsigned long long* nfail = a.nfail;
    int c[3];
    interior_coords(g, t, c);
    const long long id = lin(g, c[0], c[1], c[2]);
    const double ps = psi ? psi[id] : 1.0;
    const double al = alp ? alp[id] : 1.0;
    const double p2 = ps * ps, p4 = p2 * p2, ip2 = M ? rcp_pos(p2) : 1.0, ip4 = ip2 * ip2, ip6 = ip4 * ip2;
    CellIn ci;
    ci.gh = g.gh;
    ci.igh = g.igh;
    ci.xi = DYN ? a.xi : 0.0;
    ci.ighf = a.ighf;
    ci.xif = a.xif;
    ci.D = qb.p[0][id] * ip6;
    ci.S[0] = qb.p[1][id] * ip6 * ip2;
    ci.S[1] = qb.p[2][id] * ip6 * ip2;
    ci.S[2] = qb.p[3][id] * ip6 * ip2;
    ci.tau = qb.p[4][id] * ip6;
    double qEs[3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        qEs[i] = qb.p[5 + i][id];
        ci.Es[i] = qEs[i] * ip4;
        ci.B[i] = (CC ? bf.p[i][id] : cell_qB(g, bf.p[i], i, c)) * ip4;
    }
    const double et = eta ? eta[id] : eta_u;
    // flat: eta / (a_ii dt) with the host's reciprocal, no division
    ci.etat = a.stiff ? (M ? et * rcp_pos(al) * a.ia_dt : et * a.ia_dt) : -1.0;
    cell_derive(ci);
    double u[3];
    Eval e;
    bool atmo = false;
    // Newton start: this stage's last root plus its last change (a linear extrapolation
    // over steps, kept in FP32: it is only a start) when the history is kept, else the
    // latest primitives
    const bool hist = a.hs[0] != nullptr;
    F3 ust = {{0.0f, 0.0f, 0.0f}};
    if (a.atm && ci.D < a.d_atm) {
        atmo = true;   // (its history is left as it is)
    } else {
        bool fin = true;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            if (hist) {
                ust.x[i] = a.hs[i][id] + a.hd[i][id];
                u[i] = f2d_int(ust.x[i]);
            } else {
                u[i] = p2 * prim.p[1 + i][id];
            }
            if (!mag_below_int(u[i], kHi1e30)) fin = false;   // also NaN
        }
        if (!fin) u[0] = u[1] = u[2] = 0.0;
        if (refined && finite_int(r0) && finite_int(r1) && finite_int(r2)) {
            u[0] = r0;
            u[1] = r1;
            u[2] = r2;
        }
        // from the start, then from rest.  One copy of the iteration where it is a call of the
        // 72-register kernels (two spilled 1.8 KB, one 0.7 KB: 384^2 cold first solve on a metric
        // 605 -> 580 us); with the registers of the dynamo kernels two are faster.
        int it = -1;
#pragma unroll(DYN ? 2 : 1)
        for (int k = 0; k < 2; k++) {
            if (k == 1) {
                if (it >= 0 || !fin) break;
                u[0] = u[1] = u[2] = 0.0;
            }
            it = newton_solve<ACC>(ci, u, e, kmax, tol, a.tolf, k == 0 && hist && fin, ust, k == 0 && refined);
        }
        if (it < 0) {
            atomicAdd(nfail, 1ull);
            if (!a.atm) {
                // no atmosphere: leave the cell's primitives as they were, no stiff update (and
                // the stage's q_E theirs; a caller's own q keeps its value)
#pragma unroll
                for (int i = 0; i < 3; i++) {
                    if (R.p[0]) R.p[i][id] = 0.0;
                    if (a.stage_qE && a.qE_out.p[i]) a.qE_out.p[i][id] = p4 * p2 * prim.p[5 + i][id];
                }
                return;
            }
            atmo = true;
        }
    }
    double rho, pres;
    if (atmo) {
        // atmosphere: rest state at the floor density and pressure, E kept
        rho = rho_atm;
        pres = p_atm;
        u[0] = u[1] = u[2] = 0.0;
        e.E[0] = ci.Es[0];
        e.E[1] = ci.Es[1];
        e.E[2] = ci.Es[2];
    } else {
        const double iW = e.iW;
        rho = ci.D * iW;
        pres = (e.wt * iW - rho) * g.igh;
    }
    float f32[11], uh[3];
    implicit_f32<M>(rho, pres, u, e.E, ip2, f32);
#pragma unroll
    for (int i = 0; i < 3; i++) {
        f32[8 + i] = d2f_int(ci.B[i] * p4);
        uh[i] = d2f_int(u[i]);
    }
    implicit_store<M, ACC>(a, id, rho, pres, u, e.E, ip2, p4, qEs, f32, atmo ? nullptr : uh);
}

// the same as a call, so that its FP64 iteration takes neither registers nor
// instruction-cache room from the direct path
template <bool M, bool CC, bool ACC, bool DYN = false>
__device__ __noinline__ void implicit_general(const Dims& g, const ImpArgs& a, long long t, bool refined = false,
                                              double r0 = 0.0, double r1 = 0.0, double r2 = 0.0)
{
    implicit_solve<M, CC, ACC, DYN>(g, a, t, refined, r0, r1, r2);
}

// A mixed-precision cell at rest (emode 0 or 1) whose start is u = 0, from its FP64 residual;
// false where that does not vanish.  A short call: inline it cost the direct path of every
// other cell (512^2 vortex 41 -> 43 us per launch), and the general solve costs such a cell more
// (384^2 blast, cold, all but the edge at rest: 60 against 44).
template <bool M, bool CC>
__device__ __noinline__ bool implicit_rest(const Dims& g, const ImpArgs& a, long long t)
{
    int c[3];
    interior_coords(g, t, c);
    const long long id = lin(g, c[0], c[1], c[2]);
    const double ps = M && a.psi ? a.psi[id] : 1.0, al = M && a.alp ? a.alp[id] : 1.0;
    const double p2 = ps * ps, p4 = p2 * p2, ip2 = M ? rcp_pos(p2) : 1.0, ip4 = ip2 * ip2, ip6 = ip4 * ip2;
    // W = 1, E = (eta_t E* / (1 + eta_t)) (E held fixed: E*), w_t = (tau + D - U - D / Gamma_hat)
    // / (1 - 1 / Gamma_hat), and the residual is E x B - S
    const double et = a.eta ? a.eta[id] : a.eta_u;
    const double etat = M ? et * rcp_pos(al) * a.ia_dt : et * a.ia_dt;
    const double k = a.stiff ? etat * rcp_wide(1.0 + etat) : 1.0;   // (NaN for an infinite eta_t)
    double q[3], E[3], B[3], U2 = 0.0;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        q[i] = a.qb.p[5 + i][id];
        E[i] = k * (q[i] * ip4);
        B[i] = (CC ? a.bf.p[i][id] : cell_qB_in(g, a.bf.p[i], i, c, id)) * ip4;
        U2 += E[i] * E[i] + B[i] * B[i];
    }
    bool zero = k >= 0.0 && (!a.stiff || etat >= 0.0);   // (a negative eta_t holds E fixed too)
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const int j = (i + 1) % 3, l = (i + 2) % 3;
        if (!(E[j] * B[l] - E[l] * B[j] == a.qb.p[1 + i][id] * ip6 * ip2)) zero = false;
    }
    const double rho = a.qb.p[0][id] * ip6;
    const double wt = (a.qb.p[4][id] * ip6 + rho - 0.5 * U2 - rho * g.igh) * rcp_pos(1.0 - g.igh);
    if (!zero || !pos_int(wt)) return false;
    const double z[3] = {0.0, 0.0, 0.0}, pres = (wt - rho) * g.igh;
    const float uh[3] = {0.0f, 0.0f, 0.0f};
    float f32[11];
    implicit_f32<M>(rho, pres, z, E, ip2, f32);
#pragma unroll
    for (int i = 0; i < 3; i++) f32[8 + i] = d2f_int(B[i] * p4);
    implicit_store<M, true>(a, id, rho, pres, z, E, ip2, p4, q, f32, uh);
    return true;
}

// the dynamo form (xi != 0)
__device__ __forceinline__ bool has_dynamo(const ImpArgs& a) { return (__double_as_longlong(a.xi) << 1) != 0; }

// One cell, not of the dynamo form (which has no direct path: the callers take the general
// solve there).  The direct path takes the double-word Newton corrections from the kept start
// and accepts their root by the FP64 residual (ACC: the double-word one); atmosphere cells
// are written at once; everything else is implicit_general's.  The FP64 inputs are split
// into double-words as they are loaded and loaded again for the FP64 residual (L1 holds
// them), so that only one form is live during the corrections.
template <bool M, bool CC = false, bool ACC = false>
__device__ __forceinline__ void implicit_item(const Dims& g, const ImpArgs& a, long long t)
{
    int c[3];
    interior_coords(g, t, c);
    const long long id = lin(g, c[0], c[1], c[2]);
    const double* __restrict__ psi = M ? a.psi : nullptr;
    const double* __restrict__ alp = M ? a.alp : nullptr;
    const double ps = psi ? psi[id] : 1.0;
    const double p2 = ps * ps, p4 = p2 * p2, ip2 = M ? rcp_pos(p2) : 1.0, ip4 = ip2 * ip2, ip6 = ip4 * ip2;
    auto qE = [&](int i) { return a.qb.p[5 + i][id]; };
    auto qB = [&](int i) { return CC ? a.bf.p[i][id] : cell_qB_in(g, a.bf.p[i], i, c, id); };
    auto mul = [](double x, double f) { return M ? x * f : x; };
    const double D = mul(a.qb.p[0][id], ip6);
    if (a.atm && D < a.d_atm) {
        // atmosphere: rest state at the floor density and pressure, E kept; its history is
        // left as it is
        const double z[3] = {0.0, 0.0, 0.0};
        double q[3], Es[3];
        float f32[11];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            q[i] = qE(i);
            Es[i] = mul(q[i], ip4);
        }
        if (ACC) {
            implicit_f32<M>(a.rho_atm, a.p_atm, z, Es, ip2, f32);
#pragma unroll
            for (int i = 0; i < 3; i++) f32[8 + i] = d2f_int(mul(mul(qB(i), ip4), p4));
        }
        implicit_store<M, ACC>(a, id, a.rho_atm, a.p_atm, z, Es, ip2, p4, q, f32, nullptr);
        return;
    }
    // the start: this stage's last root plus its last change, or the latest velocity
    const bool hist = a.hs[0] != nullptr;
    dw ud[3];
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        if (hist) {
            ud[i] = dw_make(a.hs[i][id] + a.hd[i][id]);
        } else {
            ud[i] = dw_of(mul(a.prim.p[1 + i][id], p2));
        }
        if (!(fabsf(ud[i].hi) < 1e30f)) ok = false;   // also NaN
    }
    const double et = a.eta ? a.eta[id] : a.eta_u;
    // flat: eta / (a_ii dt) with the host's reciprocal, no division
    const double etat = a.stiff ? (M ? et * rcp_pos(alp ? alp[id] : 1.0) * a.ia_dt : et * a.ia_dt) : -1.0;
    const long long eb = __double_as_longlong(etat);
    const int emode = (eb >= 0 && eb <= 0x7ff0000000000000ll) || eb == (long long)0x8000000000000000ull ? 1 : 0;
    DwRoot rt;
    rt.M = 0.0f;
    bool acc;
    float B32[3];
    {
        // the derived constants in FP64 (formed in double-word arithmetic they would add to
        // the residual's error)
        CellIn ci;
        ci.D = D;
        ci.tau = mul(a.qb.p[4][id], ip6);
        ci.igh = g.igh;
        ci.etat = etat;
        ci.xi = 0.0;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            ci.S[i] = mul(mul(a.qb.p[1 + i][id], ip6), ip2);
            ci.Es[i] = mul(qE(i), ip4);
            ci.B[i] = mul(qB(i), ip4);
        }
        cell_derive(ci);
        CellDW cd = cell_dw(ci);
        cd.igh = {a.ighf, a.ighl};
#pragma unroll
        for (int i = 0; i < 3; i++) B32[i] = cd.B[i].hi;
        acc = ok && newton_refine_dw<ACC>(cd, ud, a.tolf, kDwEvals, &rt);
    }
    asm volatile("" ::: "memory");   // what follows loads its inputs anew
    double u[3], q[3];
    float f32[11], uh[3];
    if (ACC) {
        if (!acc) {
            // (a momentum scale of zero: a cell at rest, and a start of zero)
            const bool rest = ok && !(rt.M > 0.0f) && !((ud[0].hi != 0.0f) || (ud[1].hi != 0.0f) || (ud[2].hi != 0.0f));
            if (!(rest && implicit_rest<M, CC>(g, a, t)))
                implicit_general<M, CC, ACC>(g, a, t, ok, dw_to_double(ud[0]), dw_to_double(ud[1]), dw_to_double(ud[2]));
            return;
        }
        const double iW = dw_finite(dw_rcp(rt.W));
        const double rho = mul(a.qb.p[0][id], ip6) * iW, pres = (dw_finite(rt.wt) * iW - rho) * g.igh;
        double E[3];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            u[i] = dw_finite(ud[i]);
            uh[i] = d2f_int(u[i]);
            E[i] = dw_finite(rt.E[i]);
            q[i] = qE(i);
        }
        implicit_f32<M>(rho, pres, u, E, ip2, f32);
#pragma unroll
        for (int i = 0; i < 3; i++) f32[8 + i] = M ? d2f_int(mul(mul(qB(i), ip4), p4)) : B32[i];
        implicit_store<M, ACC>(a, id, rho, pres, u, E, ip2, p4, q, f32, uh);
    } else {
        double S[3], Es[3], B[3];
        const double Dn = mul(a.qb.p[0][id], ip6);
#pragma unroll
        for (int i = 0; i < 3; i++) {
            u[i] = dw_to_double(ud[i]);
            S[i] = mul(mul(a.qb.p[1 + i][id], ip6), ip2);
            q[i] = qE(i);
            Es[i] = mul(q[i], ip4);
            B[i] = mul(qB(i), ip4);
        }
        Accept e;
        evaluate_accept(Dn, mul(a.qb.p[4][id], ip6), S, Es, B, etat, g.igh, emode, u, e);
        const double fm = from_hi(max(mag_hi(e.f[0]), max(mag_hi(e.f[1]), mag_hi(e.f[2]))));
        // (every comparison is false for a NaN; a momentum scale that has left the range of FP32
        // accepts nothing, and a scale of zero, a cell at rest, accepts a residual of zero)
        if (!ok || !(rt.M < 1e30f) || !(fm <= a.tol * f2d_int(rt.M)) || !pos_int(e.wt) || !mag_below_int(e.W, kHi1e10)) {
            implicit_general<M, CC, ACC>(g, a, t, ok, u[0], u[1], u[2]);
            return;
        }
        const double rho = Dn * e.iW, pres = fma(e.wt, e.iW, -rho) * g.igh;
#pragma unroll
        for (int i = 0; i < 3; i++) uh[i] = d2f_int(u[i]);
        implicit_store<M, ACC>(a, id, rho, pres, u, e.E, ip2, p4, q, f32, uh);
    }
}

// ---------------------------------------------------------------------------
// face fluxes (Sec. 2.1, Sec. 2.5, Sec. 5 defaults): item t = D-face t
// ---------------------------------------------------------------------------

// a sign passed as a type
template <int S>
struct SignConst {
    static constexpr int value = S;
};

// the upwind edge EMF of Sec. 3.2 (Londrillo & Del Zanna 2004) with c+ = c- in each
// direction, where the four-state weights are all 1/4 and the diffusive coefficients
// c^2/2c are c/2: h_XY = alpha E_C^XY (X the A side, Y the B side), q_B^B reconstructed
// along A, q_B^A along B
template <typename T>
__device__ __forceinline__ T uct_edge(T hLL, T hLR, T hRL, T hRR, T ca, T cb, T qBbL, T qBbR, T qBaL, T qBaR)
{
    return scale_pow2<T, -2>(hLL + hLR + hRL + hRR) + (T(0.5) * ca) * (qBbR - qBbL) - (T(0.5) * cb) * (qBaR - qBaL);
}

// HLL flux at the D-face of linear index r0 (that of the cell above it) from the
// reconstructed states: prL / prR the 8 primitives (coordinate u^i and E^i), BL / BR the
// coordinate B with the two transverse components set; Bn the face's own normal q_B, psf and
// alf psi and alpha at the face (psi: whether there is one).  Writes twice the flux at r0.  prL,
// prR, BL, BR are overwritten.  FP32 (mixed precision).
//
// Eh (flat metric only, else NULL): Eh[C] set for an edge direction C != D whose
// third direction is inactive (a 1-D or 2-D grid).  Its edges then coincide with the
// D-faces, and the UCT EMF there needs only reconstructions along D of E_C and of the
// transverse q_B, which are this face's states: the face writes hat{E}_C, what emf_item
// computes from the same MC or PPM values (to round-off: the edge formula here is
// reduced for the coinciding states).
template <int D, bool M>
__device__ __forceinline__ void face_flux32(const Dims& g, float Bn, bool psi, float psf, float alf, long long r0,
                                            float* prL, float* prR, float* BL, float* BR, const FluxOut<float>& F,
                                            double* const* Eh)
{
    using T = float;
    constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
    const T pf2 = psf * psf, ipf2 = psi ? rcp_t(pf2) : T(1);
    // orthonormal-frame states at the face: u_hat = psi^2 u, E_hat = psi^2 E,
    // B_hat = psi^2 B (normal: q_B / psi^4)
    BL[D] = BR[D] = Bn * (ipf2 * ipf2);
    if (!M && Eh) {
        // C = D + 1: A = D + 2 (inactive), B = D; C = D + 2: A = D, B = D + 1 (inactive)
        // uct_edge with the inactive side's two states equal: the four-state mean is
        // the mean of the two D states, the normal field's jump across the inactive
        // side is zero, and the unit speeds leave (E_L + E_R -/+ jump of the transverse
        // q_B along D) / 2
        if (Eh[T1]) Eh[T1][r0] = to_f64(scale_pow2<T, -1>((prL[5 + T1] + prR[5 + T1]) - (BR[T2] - BL[T2])));
        if (Eh[T2]) Eh[T2][r0] = to_f64(scale_pow2<T, -1>((prL[5 + T2] + prR[5 + T2]) + (BR[T1] - BL[T1])));
    }
    if (psi) {
#pragma unroll
        for (int i = 0; i < 3; i++) {
            prL[1 + i] *= pf2;
            prR[1 + i] *= pf2;
            prL[5 + i] *= pf2;
            prR[5 + i] *= pf2;
            if (i != D) {
                BL[i] *= pf2;
                BR[i] *= pf2;
            }
        }
    }
    // HLL with c+ = c- = c = alpha sqrt(gamma^DD) = alpha / psi^2 (Sec. 2.5, maximal
    // diffusivity): (c f_L + c f_R - c^2 (q_R - q_L)) / 2c = (f_L + f_R - c (q_R - q_L)) / 2.
    // Each densitised q_v is psi^k_v times its flat-space (psi = alpha = 1) value and its
    // flux alpha psi^(k_v - 2) times, k = 6, 8, 8, 8, 6, 4, 4, 4: the HLL flux is then
    // alpha psi^(k_v - 2) times the flat-space HLL flux (unit speed) of the
    // orthonormal states.  F stores twice the flux (no 1/2 here: the update folds it).
    T gL[8], gR[8], iWL, iWR;
    face_hll_half<T, 1>(prL, BL, D, (T)g.gh, gL, iWL);
    face_hll_half<T, -1>(prR, BR, D, (T)g.gh, gR, iWR);
    const T h2 = alf * pf2, h4 = h2 * pf2, h6 = h4 * pf2;
    const long long o = r0;
#pragma unroll
    for (int v = 0; v < 8; v++) {
        const T hv = v == 0 || v == 4 ? h4 : (v < 4 ? h6 : h2);
        F.p[v][o] = (gL[v] + gR[v]) * hv;
    }
}

// Marching reconstruction along a line of cells, one quantity: the face states of the
// faces f0, f0+1, ... from one new cell per face.  MC keeps the last two cell values
// (FP32 also their difference) and the older cell's right-face state; PPM keeps the last
// two cell values, the newer one's MC slope, the interface value below it and the limited
// right edge of the cell before.  step() at face f takes cell f + AHEAD and returns the
// states of that face (between cells f-1 and f): in FP32 bitwise those of mc_face /
// ppm_face, whose slopes and interface values are the same expressions, each now
// evaluated once; in FP64 by fixed point (fixrec.cuh), MC's states as mc_face rounds
// them.  A march pushes the two cells before the one that step() takes at face
// f0 - WARM; the states of its WARM first steps are not valid yet.
template <typename T, bool P>
struct LineRec;

template <>
struct LineRec<double, false> {
    static constexpr int WARM = 1, AHEAD = 1;
    double a, b, l;
    __device__ __forceinline__ void push(double x)
    {
        a = b;
        b = x;
        l = 0.0;
    }
};

template <>
struct LineRec<float, false> {
    static constexpr int WARM = 1, AHEAD = 1;
    float a, b, d, l;
    __device__ __forceinline__ void push(float x)
    {
        a = b;
        b = x;
        d = b - a;
        l = 0.0f;
    }
    __device__ __forceinline__ void step(float x, float& L, float& R)
    {
        const float dn = x - b;
        const float hs = minmod3<float>(d, scale_pow2<float, -2>(x - a), dn);
        L = l;
        R = b - hs;
        l = b + hs;
        a = b;
        b = x;
        d = dn;
    }
};

// PPM at cell a0 by the FP64 (or FP32) sequence: fx_ppm_cell's outputs
template <typename T>
__device__ __forceinline__ void ppm_cell(T a0, T a1, T x, T s0, T ip, T& lo, T& hi, T& in, T& s1)
{
    s1 = ppm_slope<T>(a0, a1, x);
    in = ppm_iface_s<T>(a0, a1, s0, s1);
    lo = ip;
    hi = in;
    ppm_limit<T>(a0, lo, hi);
}

template <typename T>
struct LineRec<T, true> {
    static constexpr int WARM = 3, AHEAD = 2;
    T a0, a1, s0, ip, lr;   // a_f, a_f+1, slope_f, I_f-1/2, right edge_f-1
    __device__ __forceinline__ void push(T x)
    {
        a0 = a1;
        a1 = x;
        s0 = T(0);
        ip = a0;
        lr = a0;
    }
    __device__ __forceinline__ void step(T x, T& L, T& R)
    {
        T hi, in, s1;
        L = lr;
        bool done = false;
        if constexpr (sizeof(T) == 8) done = fx_ppm_cell(a0, a1, x, s0, ip, R, hi, in, s1);
        if (!done) ppm_cell<T>(a0, a1, x, s0, ip, R, hi, in, s1);
        lr = hi;
        ip = in;
        s0 = s1;
        a0 = a1;
        a1 = x;
    }
};

// one step of N marches: the states L, R at a face from the new values x.  FP64 MC runs
// the N fixed-point cells without a branch between them (their integer chains interleave)
// and then redoes by the FP64 sequence the ones that need it, if any do.
template <int N, typename T, bool P>
__device__ __forceinline__ void line_step(LineRec<T, P>* rec, const T* x, T* L, T* R)
{
    if constexpr (sizeof(T) == 8 && !P) {
        unsigned redo = 0;
        double l[N];
#pragma unroll
        for (int v = 0; v < N; v++) {
            L[v] = rec[v].l;
            if (!fx_mc_cell(rec[v].a, rec[v].b, x[v], R[v], l[v])) redo |= 1u << v;
        }
        if (redo) {
#pragma unroll
            for (int v = 0; v < N; v++)
                if (redo >> v & 1u) mc_cell_f64(rec[v].a, rec[v].b, x[v], R[v], l[v]);
        }
#pragma unroll
        for (int v = 0; v < N; v++) {
            rec[v].l = l[v];
            rec[v].a = rec[v].b;
            rec[v].b = x[v];
        }
    } else {
#pragma unroll
        for (int v = 0; v < N; v++) rec[v].step(x[v], L[v], R[v]);
    }
}

// item t of a face march along D in chunks of K: the padded coordinates c of the
// line (c[D] unset) and its faces f0 .. f1-1 (padded indices).  Chunks along D,
// x-fastest over the other directions; for D = 0 the chunks themselves run along x.
template <int D>
__device__ __forceinline__ void march_coords(const Dims& g, long long t, int* c, int& f0, int& f1)
{
    const int K = g.mk[D];
    int idx[3];
    // the chunk index along D takes the place of the D coordinate in an x-fastest box
    box_coords(t, D == 0 ? g.dq[0] : g.dv[0], D == 1 ? g.dq[1] : g.dv[1], idx);
    const int q = idx[D];
#pragma unroll
    for (int d = 0; d < 3; d++) c[d] = d == D ? 0 : g.ng[d] + idx[d];
    f0 = g.ng[D] + q * K;
    f1 = min(f0 + K, g.ng[D] + g.n[D] + 1);
}

// The same fluxes for K consecutive D-faces per thread (MC, or PPM when P): the thread
// marches along D with one LineRec per reconstructed quantity, so each new face loads
// one cell and reconstructs once (the per-face forms load four or six cells and
// compute two MC slopes, or three interface values and two parabola limits).  Items:
// chunks of K faces along D, x-fastest over the other directions (for D = 0 the chunks
// themselves run along x).  FP32 (mixed precision); FP64 is flux64_item.
template <int D, bool M, bool P>
__device__ __forceinline__ void flux32_item(const Dims& g, const PrimIn<float>& prim, const CP3& bf,
                                            const double* psi_in, const double* alp_in, const FluxOut<float>& F,
                                            double* const* Eh, long long t)
{
    using T = float;
    using Rec = LineRec<T, P>;
    const double* __restrict__ psi = M ? psi_in : nullptr;
    const double* __restrict__ alp = M ? alp_in : nullptr;
    constexpr int T1 = (D + 1) % 3, T2 = (D + 2) % 3;
    constexpr int NV = 10;   // 8 primitives and the two transverse B
    int c[3], f0, f1;
    march_coords<D>(g, t, c, f0, f1);
    // the line's cells lie at line + m st[D] (the other coordinates are interior)
    const long long sd = g.st[D];
    long long line = 0;
#pragma unroll
    for (int d = 0; d < 3; d++)
        if (d != D) line += c[d] * g.st[d];
    // the 10 reconstructed values of the cell at padded coordinate m along D (PPM's
    // stencil reaches a third ghost: ext_cell maps it); ps: psi there, in FP32
    auto load = [&](int m, T* x, T& ps) {
        const int mx = P ? ext_cell(g, D, m) : m;
        const long long mi = chk(g, line + map_cell(g, D, mx) * sd);
#pragma unroll
        for (int v = 0; v < 8; v++) x[v] = prim.p[v][mi];
        T ip6 = T(1);
        ps = T(1);
        if (psi) {
            ps = met_t<T>(psi[chk(g, line + mx * sd)]);
            const T p2 = ps * ps;
            ip6 = rcp_t(p2 * p2 * p2);
        }
        x[8] = prim.p[8 + T1][mi] * ip6;
        x[9] = prim.p[8 + T2][mi] * ip6;
    };
    Rec rec[NV];
    // the metric of the cells f - 1 and f beside the face, converted once per cell: psA, psB
    // (psN: the AHEAD newer cells, the newest last) and alA
    T psA = T(1), psB = T(1), psN[Rec::AHEAD], alA = T(1);
    {
        T w[2][NV], pw[2];
#pragma unroll
        for (int k = 0; k < 2; k++) load(f0 - Rec::WARM + Rec::AHEAD - 2 + k, w[k], pw[k]);
#pragma unroll
        for (int v = 0; v < NV; v++) {
            rec[v].push(w[0][v]);
            rec[v].push(w[1][v]);
        }
        if (P) {
            psN[0] = pw[0];
            psN[Rec::AHEAD - 1] = pw[1];
        } else {
            psB = pw[0];
            psN[0] = pw[1];
        }
    }
    if (alp) alA = met_t<T>(alp[chk(g, line + (f0 - 1) * sd)]);
    for (int f = f0 - Rec::WARM; f < f1; f++) {
        T x[NV], psx;
        load(f + Rec::AHEAD, x, psx);
        T prL[NV], prR[NV];
        line_step<NV>(rec, x, prL, prR);
        psA = psB;
        psB = psN[0];
        if (P) psN[0] = psN[Rec::AHEAD - 1];
        psN[Rec::AHEAD - 1] = psx;
        if (f < f0) continue;
        T BL[3], BR[3];
        BL[T1] = prL[8];
        BL[T2] = prL[9];
        BR[T1] = prR[8];
        BR[T2] = prR[9];
        const long long r0 = chk(g, line + f * sd);
        T psf = T(1), alf = T(1);
        if (psi) psf = T(0.5) * (psA + psB);
        if (alp) {
            const T alB = met_t<T>(alp[r0]);
            alf = T(0.5) * (alA + alB);
            alA = alB;
        }
        face_flux32<D, M>(g, (T)bf.p[D][chk(g, line + map_face(g, D, f) * sd)], psi != nullptr, psf, alf, r0, prL, prR,
                          BL, BR, F, Eh);
    }
}

// ---------------------------------------------------------------------------
// the FP64 face fluxes
// ---------------------------------------------------------------------------

// One side's half g = f + SG q of the unit-speed HLL flux in flat space, FP64, in the
// frame (n, t1, t2) of the face (the quantities of face_hll_half, which lists them).  With
//   e1 = B_t2 + SG E_t1,  e2 = SG E_t2 - B_t1   (the halves of E_t1 and E_t2)
// the Maxwell terms of each momentum half collect, since SG^2 = 1:
//   (E_t^2 + B_t^2) / 2 + SG (E x B)_n           = (e1^2 + e2^2) / 2
//   -E_n E_t1 - B_n B_t1 + SG (E x B)_t1         = -SG E_n e1 + B_n e2
//   -E_n E_t2 - B_n B_t2 + SG (E x B)_t2         = -SG E_n e2 - B_n e1
// so that with a = u_n + SG W, N = (E_n^2 + B_n^2) / 2 and Q = (e1^2 + e2^2) / 2
//   S_n: rho h a u_n + Q + (p - N),   tau: a (rho h W - rho) + SG (Q - (p - N)).
// 30 FP64 instructions where the separate terms took 45.  W = s (1 + e/2 + 3 e^2 / 8) from
// an FP32 estimate y of 1/sqrt(x): s = x y, e = 1 - s y (as in rsqrt_ge1).
// st: rho, u_n, u_t1, u_t2, p, E_n, E_t1, E_t2; Bt: B_t1, B_t2; hBn2 = B_n^2 / 2.
template <int SG>
__device__ __forceinline__ void hll_half64(const double* st, const double* Bt, double Bn, double hBn2, double gh,
                                           double* g, double& W)
{
    constexpr double sg = SG;
    const double rho = st[0], u0 = st[1], u1 = st[2], u2 = st[3], p = st[4], En = st[5];
    const double x = fma(u0, u0, fma(u1, u1, fma(u2, u2, 1.0)));
    const double y = f2d_int(rsqrtf(d2f_int(x)));
    const double s = x * y, e = fma(-s, y, 1.0);
    W = fma(s, e * fma(0.375, e, 0.5), s);
    if (!mag_below_int(x, kHi2p127)) W = x * rsqrt(x);   // the estimate has left the range of FP32
    const double h = fma(gh, p, rho), hW = h * W;
    const double e1 = SG > 0 ? Bt[1] + st[6] : Bt[1] - st[6];
    const double e2 = SG > 0 ? st[7] - Bt[0] : -st[7] - Bt[0];
    const double Q2 = fma(e1, e1, e2 * e2);
    const double pm = fma(-0.5 * En, En, p - hBn2);
    const double a = SG > 0 ? u0 + W : u0 - W;
    const double K = h * a;
    g[0] = rho * a;
    g[1] = fma(K, u0, fma(0.5, Q2, pm));
    g[2] = fma(K, u1, fma(-sg * En, e1, Bn * e2));
    g[3] = fma(K, u2, fma(-sg * En, e2, -Bn * e1));
    g[4] = fma(a, hW - rho, SG > 0 ? fma(0.5, Q2, -pm) : fma(-0.5, Q2, pm));
    g[5] = sg * En;
    g[6] = e1;
    g[7] = e2;
}

// Threads per block of the kernels that run flux64_item, and the shared doubles it takes
// (SL per thread and quantity: MC a, b, lo, hi; PPM a0, a1, s0, ip, lo, hi).  us per stencil
// launch by threads per block and least blocks per SM: MC 512^2 128 x 4 116.5, 128 x 5 117.1,
// 96 x 5 121.1, 64 x 8 117.6; PPM 301^2 96 x 4 159.1, 64 x 6 155.1, 64 x 7 166.5, 32 x 14 167.9.
template <bool P, bool CC>
struct Flux64 {
    static constexpr int NV = CC ? 12 : 10;        // 8 primitives, B_t1, B_t2 (CC: B_n, B_t1, B_t2, Phi)
    static constexpr int SL = P ? 6 : 4;
    static constexpr int NT = P ? 64 : 128;
    static constexpr int SM = NV * SL * NT;        // at most 48 KB
    // a march's start-up in faces (march_len): PPM reconstructs two cells before the first face
    // and loads four, which are two faces' work here, where reconstruction bounds the kernel
    // (at 1, as in FP32, star 96^3 took marches too short: 4.22 ms per launch, 3.70 at 2 or 3; 24^3
    // to 64^3 and the 2-D vortices the same at 1, 2 and 3)
    static constexpr double C0 = P ? 2.0 : 0.6;
};

// The FP64 fluxes of K consecutive d-faces per thread, marched along d; CC: the 12
// variables of the GLM scheme (cell-centred q_B in bq, q_Phi).
//
// A thread goes from cell to cell: it reconstructs the cell's two edge states, forms the
// right state's half of the HLL flux at the lower face and completes that face, then the
// left state's half at the upper face, which it carries to the next cell.  The cell
// windows and edge states of the NV quantities lie in the thread's column of shared
// memory, so that the reconstruction is a short rolled loop: held in registers it was
// unrolled NV-fold, which took 168 registers (three blocks per SM) and a loop body beyond
// the instruction cache (a fifth of the stalls were instruction fetches).  The direction
// is a run-time value (the components are permuted as they are loaded), so that the tasks
// of a launch share one code.
//
// Eh (flat metric, CT; NULL or with NULL entries): the edge EMFs along the directions
// C != d whose third direction is inactive (1-D and 2-D grids).  Those edges coincide
// with the d-faces, and uct_edge with the inactive side's two states equal and unit
// speeds leaves (E_L + E_R -/+ the jump of the transverse q_B along d) / 2, which is half
// the difference of the two HLL halves of E_C.
template <bool M, bool P, bool CC>
__device__ __forceinline__ void flux64_item(const Dims& g, int d, const double* const* prim, const double* const* bq,
                                            const double* __restrict__ qphi, const double* psi_in,
                                            const double* alp_in, double* const* F, double* const* vbar,
                                            double* const* Eh, double* sm, long long t)
{
    using C = Flux64<P, CC>;
    constexpr int NV = C::NV, SL = C::SL, NT = C::NT, G = CC ? 4 : 5;   // quantities in groups of G
    constexpr int LO = SL - 2, HI = SL - 1;
    constexpr int NF = CC ? 12 : 8;
    const double* __restrict__ psi = M ? psi_in : nullptr;
    const double* __restrict__ alp = M ? alp_in : nullptr;
    double* const col = sm + threadIdx.x;
    const int t1 = d == 2 ? 0 : d + 1, t2 = d == 0 ? 2 : d - 1;
    // the line's chunk of faces f0 .. f1-1 and the offset of its cells at d-coordinate 0
    int idx[3];
    box_coords(t, d == 0 ? g.dq[0] : g.dv[0], d == 1 ? g.dq[1] : g.dv[1], idx);
    const int q0 = d == 0 ? idx[0] : (d == 1 ? idx[1] : idx[2]);
    const int f0 = g.ng[d] + q0 * g.mk[d], f1 = min(f0 + g.mk[d], g.ng[d] + g.n[d] + 1);
    long long line = 0;
    long long up[2] = {0, 0};   // from a cell's lower t1 / t2 face to its upper one
#pragma unroll
    for (int e = 0; e < 3; e++) {
        if (e == d) continue;
        const int ce = g.ng[e] + idx[e];
        line += ce * g.st[e];
        const int he = g.bc[e] == BC_PERIODIC && ce + 1 == g.ng[e] + g.n[e] ? g.ng[e] : ce + 1;
        if (g.act[e]) up[e == t1 ? 0 : 1] = (he - ce) * g.st[e];
    }
    const long long sd = g.st[d];
    // psi^2 and alpha at the face carried along, its normal B, and the left state's halves
    double pf2 = 1.0, alf = 1.0, Bn = 0.0, hBn2 = 0.0, gL[NF], vL[2] = {0.0, 0.0};
#pragma unroll
    for (int v = 0; v < NF; v++) gL[v] = 0.0;
    // one side's half flux at the carried face from the edge states in `slot`
    auto half = [&](int slot, auto sgc, double* gh, double* vh) {
        constexpr int SG = decltype(sgc)::value;
        double pr[8], B[3], W;   // B: n, t1, t2
#pragma unroll
        for (int v = 0; v < 8; v++) pr[v] = col[(v * SL + slot) * NT];
        if (CC) {
#pragma unroll
            for (int e = 0; e < 3; e++) B[e] = col[((8 + e) * SL + slot) * NT];
        } else {
            B[0] = Bn;
            B[1] = col[(8 * SL + slot) * NT];
            B[2] = col[(9 * SL + slot) * NT];
        }
        if (psi) {
            // orthonormal frame: u_hat = psi^2 u, E_hat = psi^2 E, B_hat = psi^2 B
#pragma unroll
            for (int i = 0; i < 3; i++) {
                pr[1 + i] *= pf2;
                pr[5 + i] *= pf2;
                if (CC || i > 0) B[i] *= pf2;
            }
        }
        if (CC) hBn2 = 0.5 * B[0] * B[0];
        hll_half64<SG>(pr, B + 1, B[0], hBn2, g.gh, gh, W);
        if (CC) {
            // unit-speed halves of q_B (f_B^j = eta^{jnk} E_k) and of q_Phi (f = B^n)
            gh[8] = SG * B[0];
            gh[9] = SG * B[1] - pr[7];
            gh[10] = SG * B[2] + pr[6];
            gh[11] = B[0] + SG * col[(11 * SL + slot) * NT];
        }
        if (vbar && vbar[0]) {
            const double iW = rcp_wide(W);
            vh[0] = pr[2] * iW;
            vh[1] = pr[3] * iW;
        }
    };
    // centre cell m takes cell m + AHEAD; the first cells fill the windows
    constexpr int AHEAD = P ? 2 : 1, WARM = P ? 2 : 0;
    for (int m = f0 - 3 - WARM; m < f1; m++) {
        const int mx = P ? ext_cell(g, d, m + AHEAD) : m + AHEAD;
        const long long mi = chk(g, line + map_cell(g, d, mx) * sd);
        double ip6 = 1.0;
        if (psi) {
            const double ps = psi[chk(g, line + mx * sd)], p2 = ps * ps;
            ip6 = rcp_pos(p2 * p2 * p2);
        }
#pragma unroll 1
        for (int q = 0; q < NV / G; q++) {
            double x[G];
            if (CC) {
                if (q == 0) {
                    x[0] = prim[0][mi];
                    x[1] = prim[1 + d][mi];
                    x[2] = prim[1 + t1][mi];
                    x[3] = prim[1 + t2][mi];
                } else if (q == 1) {
                    x[0] = prim[4][mi];
                    x[1] = prim[5 + d][mi];
                    x[2] = prim[5 + t1][mi];
                    x[3] = prim[5 + t2][mi];
                } else {
                    x[0] = bq[d][mi] * ip6;
                    x[1] = bq[t1][mi] * ip6;
                    x[2] = bq[t2][mi] * ip6;
                    x[3] = qphi[mi] * ip6;
                }
            } else if (q == 0) {
                x[0] = prim[0][mi];
                x[1] = prim[1 + d][mi];
                x[2] = prim[1 + t1][mi];
                x[3] = prim[1 + t2][mi];
                x[G - 1] = prim[4][mi];
            } else {
                x[0] = prim[5 + d][mi];
                x[1] = prim[5 + t1][mi];
                x[2] = prim[5 + t2][mi];
                // the mean of the cell's two faces (an inactive direction: the cell value twice)
                x[3] = scale_pow2<double, -1>(bq[t1][mi] + bq[t1][chk(g, mi + up[0])]) * ip6;
                x[G - 1] = scale_pow2<double, -1>(bq[t2][mi] + bq[t2][chk(g, mi + up[1])]) * ip6;
            }
            double* const w = col + q * (G * SL * NT);
            if (m < f0 - 1 - WARM) {
#pragma unroll
                for (int i = 0; i < G; i++) {
                    double* const s = w + i * (SL * NT);
                    s[0] = s[NT];
                    s[NT] = x[i];
                    if (P) {
                        s[2 * NT] = 0.0;
                        s[3 * NT] = x[i];
                    }
                }
                continue;
            }
            unsigned redo = 0;
#pragma unroll
            for (int i = 0; i < G; i++) {
                double* const s = w + i * (SL * NT);
                double lo, hi;
                if (P) {
                    double in, s1;
                    if (!fx_ppm_cell(s[0], s[NT], x[i], s[2 * NT], s[3 * NT], lo, hi, in, s1))
                        ppm_cell<double>(s[0], s[NT], x[i], s[2 * NT], s[3 * NT], lo, hi, in, s1);
                    s[0] = s[NT];
                    s[NT] = x[i];
                    s[2 * NT] = s1;
                    s[3 * NT] = in;
                } else {
                    if (!fx_mc_cell(s[0], s[NT], x[i], lo, hi)) redo |= 1u << i;
                }
                s[LO * NT] = lo;
                s[HI * NT] = hi;
            }
            if (!P) {
                if (redo) {
#pragma unroll 1
                    for (int i = 0; i < G; i++) {
                        double* const s = w + i * (SL * NT);
                        double xi = x[0];
#pragma unroll
                        for (int j = 1; j < G; j++)
                            if (i == j) xi = x[j];
                        if (redo >> i & 1u) mc_cell_f64(s[0], s[NT], xi, s[LO * NT], s[HI * NT]);
                    }
                }
#pragma unroll
                for (int i = 0; i < G; i++) {
                    double* const s = w + i * (SL * NT);
                    s[0] = s[NT];
                    s[NT] = x[i];
                }
            }
        }
        if (m < f0 - 1) continue;
        const long long r0 = chk(g, line + m * sd);
        if (m >= f0) {
            // HLL with c+ = c- = c = alpha sqrt(gamma^nn) = alpha / psi^2 (Sec. 2.5, maximal
            // diffusivity): (c f_L + c f_R - c^2 (q_R - q_L)) / 2c = (f_L + f_R - c (q_R -
            // q_L)) / 2.  Each densitised q_v is psi^k_v times its flat-space (psi = alpha = 1)
            // value and its flux alpha psi^(k_v - 2) times, k = 6, 8, 8, 8, 6, 4, 4, 4 (GLM:
            // and 4, 4, 4, 6): the HLL flux is then alpha psi^(k_v - 2) times the flat-space
            // HLL flux (unit speed) of the orthonormal states.  F stores twice the flux (the
            // update folds the 1/2).
            double gR[NF], vR[2];
            half(LO, SignConst<-1>(), gR, vR);
            const double h2 = alf * pf2, h4 = h2 * pf2, h6 = h4 * pf2;
            const int o[NF > 8 ? 12 : 8] = {0, 1 + d, 1 + t1, 1 + t2, 4, 5 + d, 5 + t1, 5 + t2};
#pragma unroll
            for (int v = 0; v < NF; v++) {
                const double hv = v == 0 || v == 4 || v == 11 ? h4 : (v < 4 ? h6 : h2);
                const int ov = v < 8 ? o[v < 8 ? v : 0] : (v == 8 ? 8 + d : (v == 9 ? 8 + t1 : (v == 10 ? 8 + t2 : 11)));
                F[ov][r0] = (gL[v] + gR[v]) * hv;
            }
            if (!M && !CC && Eh) {
                if (Eh[t1]) Eh[t1][r0] = scale_pow2<double, -1>(gL[6] - gR[6]);
                if (Eh[t2]) Eh[t2][r0] = scale_pow2<double, -1>(gL[7] - gR[7]);
            }
            if (vbar && vbar[0]) {
                // App. A steps (i)-(ii): vhat^j = alpha v^j (beta = 0) of the L and R states,
                // vbar^j = (c- vhat^j_R + c+ vhat^j_L)/(c- + c+), their mean for c+ = c-;
                // v^j = u_hat^j / (psi^2 W)
                const double al = 0.5 * alf * (psi ? rcp_pos(pf2) : 1.0);
                vbar[0][r0] = al * (vL[0] + vR[0]);
                vbar[1][r0] = al * (vL[1] + vR[1]);
            }
        }
        if (m + 1 < f1) {
            const long long r1 = chk(g, r0 + sd);
            const double psf = psi ? mean2<double>(psi[r0], psi[r1]) : 1.0;
            alf = alp ? mean2<double>(alp[r0], alp[r1]) : 1.0;
            pf2 = psf * psf;
            if (!CC) {
                Bn = bq[d][chk(g, line + map_face(g, d, m + 1) * sd)];   // B_hat: q_B / psi^4
                if (psi) {
                    const double i2 = rcp_pos(pf2);
                    Bn *= i2 * i2;
                }
                hBn2 = 0.5 * Bn * Bn;
            }
            half(HI, SignConst<1>(), gL, vL);
        }
    }
}

// ---------------------------------------------------------------------------
// upwind constrained transport (Sec. 3.2): item t = C-edge t
// ---------------------------------------------------------------------------

// Face speeds at a C-edge (Sec. 2.5: c = alpha sqrt(gamma^dd) = alpha / psi^2 at a face,
// whose alpha and psi are the means of the two cells beside it): cab[0] the larger of
// the (up to two) A-faces touching the edge, cab[1] likewise for the B-faces; 1 in an
// inactive direction.  The larger of a0/q0 and a1/q1 is picked by comparing a0 q1 with
// a1 q0, and both quotients come from one reciprocal.
template <typename T>
__device__ __forceinline__ void edge_speeds(const Dims& g, const double* __restrict__ psi,
                                            const double* __restrict__ alp, long long i0, bool aa, bool ba,
                                            long long sA, long long sB, T* cab)
{
    T num[2] = {T(1), T(1)}, den[2] = {T(1), T(1)};
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const bool act = k == 0 ? aa : ba, oth = k == 0 ? ba : aa;
        if (!act) continue;
        const long long sn = k == 0 ? sA : sB, so = k == 0 ? sB : sA;
        for (int tt = 0; tt < (oth ? 2 : 1); tt++) {
            const long long cf = chk(g, i0 - tt * so), cfm = chk(g, cf - sn);
            const T psf = psi ? mean2<T>(psi[cfm], psi[cf]) : T(1);
            const T alf = alp ? mean2<T>(alp[cfm], alp[cf]) : T(1);
            const T q = psf * psf;
            if (tt == 0 || alf * den[k] > num[k] * q) {
                num[k] = alf;
                den[k] = q;
            }
        }
    }
    const T r = rcp_t(den[0] * den[1]);
    cab[0] = num[0] * den[1] * r;
    cab[1] = num[1] * den[0] * r;
}

// P: PPM reconstruction (six cells or faces per pass) instead of MC (four)
template <int C, bool M, typename T, bool P = false>
__device__ __forceinline__ void emf_item(const Dims& g, const PrimIn<T>& prim, const CP3& bf, const double* psi_in,
                                         const double* alp_in, double* __restrict__ Eh, long long t)
{
    constexpr int NS = P ? 6 : 4, OFF = P ? 3 : 2;
    const double* __restrict__ psi = M ? psi_in : nullptr;
    const double* __restrict__ alp = M ? alp_in : nullptr;
    constexpr int A = (C + 1) % 3, B = (C + 2) % 3;
    const bool aa = g.act[A], ba = g.act[B];
    const T* __restrict__ Ec = prim.p[5 + C];
    // edges: n[d] along C, n[d] + 1 along an active transverse d (1 if inactive)
    int c[3];
    box_coords(t, C == 0 ? g.dv[0] : g.dvp[0], C == 1 ? g.dv[1] : g.dvp[1], c);
#pragma unroll
    for (int d = 0; d < 3; d++) c[d] += g.ng[d];
    // steps (ii)-(iii): covariant E_C = psi^4 E^C, to A-faces then along B
    T s[2][NS];   // [X = A-side L/R][B offset -OFF..+OFF-1]
    const int nb = ba ? NS : 1;
    for (int ob = 0; ob < nb; ob++) {
        int cb[3] = {c[0], c[1], c[2]};
        if (ba) cb[B] = P ? ext_cell(g, B, c[B] + ob - OFF) : c[B] + ob - OFF;
        if (aa) {
            T v[NS];
#pragma unroll
            for (int sa = 0; sa < NS; sa++) {
                int cs[3] = {cb[0], cb[1], cb[2]};
                cs[A] = P ? ext_cell(g, A, cb[A] + sa - OFF) : cb[A] + sa - OFF;
                const T ps = psi ? met_t<T>(psi[lin(g, cs[0], cs[1], cs[2])]) : T(1);
                const T p2 = ps * ps;
                v[sa] = p2 * p2 * Ec[cell_at(g, cs)];
            }
            if (P) ppm_face<T>(v, s[0][ob], s[1][ob]);
            else mc_face<T>(v[0], v[1], v[2], v[NS - 1], s[0][ob], s[1][ob]);
        } else {
            const T ps = psi ? met_t<T>(psi[lin(g, cb[0], cb[1], cb[2])]) : T(1);
            const T p2 = ps * ps;
            s[0][ob] = s[1][ob] = p2 * p2 * Ec[cell_at(g, cb)];
        }
    }
    T EXY[2][2];
#pragma unroll
    for (int X = 0; X < 2; X++) {
        if (!ba) EXY[X][0] = EXY[X][1] = s[X][0];
        else if (P) ppm_face<T>(s[X], EXY[X][0], EXY[X][1]);
        else mc_face<T>(s[X][0], s[X][1], s[X][2], s[X][NS - 1], EXY[X][0], EXY[X][1]);
    }
    // step (iv): q_B^B (B-faces) along A, q_B^A (A-faces) along B
    T qBbL, qBbR, qBaL, qBaR;
    if (aa) {
        T v[NS];
#pragma unroll
        for (int sa = 0; sa < NS; sa++) {
            int cs[3] = {c[0], c[1], c[2]};
            cs[A] = P ? ext_cell(g, A, c[A] + sa - OFF) : c[A] + sa - OFF;
            v[sa] = (T)bf.p[B][face_at(g, B, cs)];
        }
        if (P) ppm_face<T>(v, qBbL, qBbR);
        else mc_face<T>(v[0], v[1], v[2], v[NS - 1], qBbL, qBbR);
    } else {
        qBbL = qBbR = (T)bf.p[B][face_at(g, B, c)];
    }
    if (ba) {
        T v[NS];
#pragma unroll
        for (int sb = 0; sb < NS; sb++) {
            int cs[3] = {c[0], c[1], c[2]};
            cs[B] = P ? ext_cell(g, B, c[B] + sb - OFF) : c[B] + sb - OFF;
            v[sb] = (T)bf.p[A][face_at(g, A, cs)];
        }
        if (P) ppm_face<T>(v, qBaL, qBaR);
        else mc_face<T>(v[0], v[1], v[2], v[NS - 1], qBaL, qBaR);
    } else {
        qBaL = qBaR = (T)bf.p[A][face_at(g, A, c)];
    }
    // lapse at the edge (mean of the adjacent cells) and the face speeds
    const long long i0 = lin(g, c[0], c[1], c[2]);
    const long long sA = aa ? g.st[A] : 0, sB = ba ? g.st[B] : 0;
    T ale = T(1), ca = T(1), cb = T(1);
    if (alp || psi) {
        // mean of the 1, 2 or 4 cells around the edge
        T sum = alp ? met_t<T>(alp[i0]) : T(1), w = T(1);
        if (aa) { sum += alp ? met_t<T>(alp[chk(g, i0 - sA)]) : T(1); w = T(0.5); }
        if (ba) {
            sum += alp ? met_t<T>(alp[chk(g, i0 - sB)]) : T(1);
            if (aa) sum += alp ? met_t<T>(alp[chk(g, i0 - sA - sB)]) : T(1);
            w *= T(0.5);
        }
        ale = sum * w;
        T cab[2];
        edge_speeds<T>(g, psi, alp, i0, aa, ba, sA, sB, cab);
        ca = cab[0];
        cb = cab[1];
    }
    // steps (v)-(vii): hat{E}^{XY} = alpha E_C^{XY}; Londrillo & Del Zanna (2004) with
    // c+ = c- in each direction, where the four-state weights are all 1/4 and the
    // diffusive coefficients c^2/2c are c/2
    const T hLL = ale * EXY[0][0], hLR = ale * EXY[0][1], hRL = ale * EXY[1][0], hRR = ale * EXY[1][1];
    Eh[i0] = to_f64(uct_edge<T>(hLL, hLR, hRL, hRR, ca, cb, qBbL, qBbR, qBaL, qBaR));
}

// The metric of a C-edge among the four cells c00, cA (one below along A), cB and cAB: the
// lapse there (their mean) and half the larger of the two A-face speeds alpha / psi^2 and
// of the two B-face ones (alpha and psi at a face: the means of its two cells).  The larger
// is picked in FP32 where that decides (the two differ by more than its rounding), else by
// cross-multiplying in FP64, so that FP64 forms one speed per direction, not two; both come
// from one reciprocal.
__device__ __forceinline__ void edge_metric64(const double* __restrict__ psi, const double* __restrict__ alp,
                                              long long c00, long long cA, long long cB, long long cAB, double& ale,
                                              double& ha, double& hb)
{
    const double p00 = psi ? psi[c00] : 1.0, pA = psi ? psi[cA] : 1.0, pB = psi ? psi[cB] : 1.0,
                 pAB = psi ? psi[cAB] : 1.0;
    const double a00 = alp ? alp[c00] : 1.0, aA = alp ? alp[cA] : 1.0, aB = alp ? alp[cB] : 1.0,
                 aAB = alp ? alp[cAB] : 1.0;
    const double sA0 = a00 + aA, sA1 = aB + aAB;   // twice alpha at the A-faces of the two rows
    ale = scale_pow2<double, -2>(sA0 + sA1);
    const float f00 = d2f_int(p00), fA = d2f_int(pA), fB = d2f_int(pB), fAB = d2f_int(pAB);
    const float g00 = d2f_int(a00), gA = d2f_int(aA), gB = d2f_int(aB), gAB = d2f_int(aAB);
    double num[2], den[2];   // speed = 2 num / den with num = twice alpha, den = (twice psi)^2
#pragma unroll
    for (int k = 0; k < 2; k++) {
        // face 0: cells c00 and cA (k = 0) or cB (k = 1); face 1: the other two
        const float h0 = f00 + (k == 0 ? fA : fB), h1 = (k == 0 ? fB : fA) + fAB;
        const float x0 = (g00 + (k == 0 ? gA : gB)) * h1 * h1, x1 = ((k == 0 ? gB : gA) + gAB) * h0 * h0;
        bool second = x1 > x0;
        if (!(fabsf(x0 - x1) > 4e-6f * x0)) {
            const double q0 = p00 + (k == 0 ? pA : pB), q1 = (k == 0 ? pB : pA) + pAB;
            const double n0 = k == 0 ? sA0 : a00 + aB, n1 = k == 0 ? sA1 : aA + aAB;
            second = n1 * (q0 * q0) > n0 * (q1 * q1);
        }
        const double u = second ? (k == 0 ? pB : pA) : p00, v = second ? pAB : (k == 0 ? pA : pB);
        const double q = u + v;
        den[k] = q * q;
        num[k] = k == 0 ? (second ? sA1 : sA0) : (second ? aA : a00) + (second ? aAB : aB);
    }
    const double r = rcp_pos(den[0] * den[1]);
    ha = num[0] * (den[1] * r);
    hb = num[1] * (den[0] * r);
}

// The EMFs of K consecutive C-edges along B per thread (MC, or PPM when P; A and B both
// active): the A-direction reconstruction of E_C on each row of cells along B, and q_B^A,
// are marched along B with LineRec (one new row per edge instead of four or six), so each
// edge computes one A-row, three one-cell B steps and its own q_B^B reconstruction, with the
// sums of emf_item (in FP32 bitwise).  Items: chunks of K edges along B, x-fastest over the
// other two directions (the chunks run along x when B = 0).  C is a run-time value (the tasks
// of a launch share one code) and the line's offsets are formed once.
template <bool M, typename T, bool P>
__device__ __forceinline__ void emf_line_item(const Dims& g, int C, const T* const* prim, const double* const* bf,
                                              const double* psi_in, const double* alp_in, double* __restrict__ Eh,
                                              long long t)
{
    using Rec = LineRec<T, P>;
    constexpr int NS = P ? 6 : 4, OFF = P ? 3 : 2;
    const double* __restrict__ psi = M ? psi_in : nullptr;
    const double* __restrict__ alp = M ? alp_in : nullptr;
    const int A = C == 2 ? 0 : C + 1, B = C == 0 ? 2 : C - 1;
    const T* __restrict__ Ec = prim[5 + C];
    const double* __restrict__ qA = bf[A];
    const double* __restrict__ qB = bf[B];
    // x-fastest box: the chunks along B, n[C] edges along C, n[A] + 1 along A
    int idx[3];
    box_coords(t, B == 0 ? g.dq[0] : (C == 0 ? g.dv[0] : g.dvp[0]), B == 1 ? g.dq[1] : (C == 1 ? g.dv[1] : g.dvp[1]),
               idx);
    auto at = [&](int d) { return d == 0 ? idx[0] : (d == 1 ? idx[1] : idx[2]); };
    const int f0 = g.ng[B] + at(B) * g.mk[B], f1 = min(f0 + g.mk[B], g.ng[B] + g.n[B] + 1);
    const int cA = g.ng[A] + at(A);
    const long long line = (g.ng[C] + at(C)) * g.st[C], sA = g.st[A], sB = g.st[B];
    // the cells along A around the edge (mapped, and where the metric is read), its A-face
    long long ia[NS], pa[NS];
#pragma unroll
    for (int k = 0; k < NS; k++) {
        const int m = P ? ext_cell(g, A, cA + k - OFF) : cA + k - OFF;
        ia[k] = line + map_cell(g, A, m) * sA;
        pa[k] = line + m * sA;
    }
    const long long fa = line + map_face(g, A, cA) * sA;
    auto recA = [&](const T* v, T& L, T& R) {
        if (P) ppm_face<T>(v, L, R);
        else mc_face<T>(v[0], v[1], v[2], v[NS - 1], L, R);
    };
    Rec rec[3];
#pragma unroll
    for (int v = 0; v < 3; v++) {
        rec[v].push(T(0));
        rec[v].push(T(0));
    }
    for (int f = f0 - Rec::WARM - 2; f < f1; f++) {
        // row f + AHEAD along B: covariant E_C = psi^4 E^C reconstructed along A to the
        // A-face, and q_B^A at that A-face
        const int mb = P ? ext_cell(g, B, f + Rec::AHEAD) : f + Rec::AHEAD;
        const long long rb = map_cell(g, B, mb) * sB;
        T x3[3];
        {
            T v[NS];
            if constexpr (sizeof(T) == 8) {
#pragma unroll
                for (int k = 0; k < NS; k++) {
                    v[k] = Ec[chk(g, ia[k] + rb)];
                    if (psi) {
                        const T ps = psi[chk(g, pa[k] + mb * sB)], p2 = ps * ps;
                        v[k] *= p2 * p2;
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < NS; k++) {
                    const T ps = psi ? met_t<T>(psi[chk(g, pa[k] + mb * sB)]) : T(1);
                    const T p2 = ps * ps;
                    v[k] = p2 * p2 * Ec[chk(g, ia[k] + rb)];
                }
            }
            recA(v, x3[0], x3[1]);
        }
        x3[2] = (T)qA[chk(g, fa + rb)];
        if (f < f0 - Rec::WARM) {
#pragma unroll
            for (int v = 0; v < 3; v++) rec[v].push(x3[v]);
            continue;
        }
        T L[3], R[3];
        line_step<3>(rec, x3, L, R);
        if (f < f0) continue;
        // q_B^B (B-faces) along A
        T qL, qR;
        {
            const long long jb = map_face(g, B, f) * sB;
            T v[NS];
#pragma unroll
            for (int k = 0; k < NS; k++) v[k] = (T)qB[chk(g, ia[k] + jb)];
            recA(v, qL, qR);
        }
        const long long i0 = chk(g, line + cA * sA + f * sB);
        if constexpr (sizeof(T) == 8) {
            // uct_edge: the mean of the four states times the edge's lapse, and half the larger
            // face speed of each direction times the jump of q_B
            const double mean = scale_pow2<double, -2>((L[0] + R[0]) + (L[1] + R[1]));
            if (alp || psi) {
                double ale, ha, hb;
                edge_metric64(psi, alp, i0, chk(g, i0 - sA), chk(g, i0 - sB), chk(g, i0 - sA - sB), ale, ha, hb);
                Eh[i0] = fma(-hb, R[2] - L[2], fma(ha, qR - qL, ale * mean));
            } else {
                Eh[i0] = fma(-0.5, R[2] - L[2], fma(0.5, qR - qL, mean));
            }
        } else {
            T ale = T(1), cab[2] = {T(1), T(1)};
            if (alp || psi) {
                T sum = alp ? met_t<T>(alp[i0]) : T(1);
                sum += alp ? met_t<T>(alp[chk(g, i0 - sA)]) : T(1);
                sum += alp ? met_t<T>(alp[chk(g, i0 - sB)]) : T(1);
                sum += alp ? met_t<T>(alp[chk(g, i0 - sA - sB)]) : T(1);
                ale = sum * T(0.25);
                edge_speeds<T>(g, psi, alp, i0, true, true, sA, sB, cab);
            }
            Eh[i0] = to_f64(uct_edge<T>(ale * L[0], ale * R[0], ale * L[1], ale * R[1], cab[0], cab[1], qL, qR, L[2],
                                        R[2]));
        }
    }
}

// ---------------------------------------------------------------------------
// ideal-limit edge EMF (App. A), FP64: item t = C-edge t (as emf_item)
// ---------------------------------------------------------------------------

// transport velocity vhat^j = alpha v^j of the cell at padded coordinates cs (the
// "face" value in an inactive direction)
__device__ __forceinline__ double cell_vhat(const Dims& g, const CP8& prim, const double* __restrict__ psi,
                                            const double* __restrict__ alp, int j, const int* cs)
{
    const long long mi = cell_at(g, cs), ri = lin(g, cs[0], cs[1], cs[2]);
    const double ps = psi ? psi[ri] : 1.0;
    const double p4 = ps * ps * ps * ps;
    const double u0 = prim.p[1][mi], u1 = prim.p[2][mi], u2 = prim.p[3][mi];
    return (alp ? alp[ri] : 1.0) * prim.p[1 + j][mi] * rsqrt(1.0 + p4 * (u0 * u0 + u1 * u1 + u2 * u2));
}

// vb[d][k]: transport velocities at the d-faces, component (d + 1 + k) % 3
template <int C, bool M>
__device__ __forceinline__ void emf_ideal_item(const Dims& g, const CP8& prim, const CP3& bf, const double* psi_in,
                                               const double* alp_in, const double* const (*vb)[2],
                                               double* __restrict__ Eh, long long t)
{
    const double* __restrict__ psi = M ? psi_in : nullptr;
    const double* __restrict__ alp = M ? alp_in : nullptr;
    constexpr int A = (C + 1) % 3, B = (C + 2) % 3;
    const bool aa = g.act[A], ba = g.act[B];
    // edges: n[d] along C, n[d] + 1 along an active transverse d (1 if inactive)
    int c[3];
    box_coords(t, C == 0 ? g.dv[0] : g.dvp[0], C == 1 ? g.dv[1] : g.dvp[1], c);
#pragma unroll
    for (int d = 0; d < 3; d++) c[d] += g.ng[d];
    // step (iii): q_B^B and vbar^A (both at B-faces) along A; q_B^A and vbar^B (A-faces)
    // along B.  vbar^A is component A = B + 2 of the B-faces, vbar^B component B = A + 1
    // of the A-faces.
    double qBbL, qBbR, qBaL, qBaR, vaL, vaR, vbL, vbR;
    {
        double q[4], v[4];
        const int ns = aa ? 4 : 1;
        for (int sa = 0; sa < ns; sa++) {
            int cs[3] = {c[0], c[1], c[2]};
            if (aa) cs[A] += sa - 2;
            const long long fi = face_at(g, B, cs);
            q[sa] = bf.p[B][fi];
            v[sa] = ba ? vb[B][1][fi] : cell_vhat(g, prim, psi, alp, A, cs);
        }
        if (aa) {
            mc_face<double>(q[0], q[1], q[2], q[3], qBbL, qBbR);
            mc_face<double>(v[0], v[1], v[2], v[3], vaL, vaR);
        } else {
            qBbL = qBbR = q[0];
            vaL = vaR = v[0];
        }
    }
    {
        double q[4], v[4];
        const int ns = ba ? 4 : 1;
        for (int sb = 0; sb < ns; sb++) {
            int cs[3] = {c[0], c[1], c[2]};
            if (ba) cs[B] += sb - 2;
            const long long fi = face_at(g, A, cs);
            q[sb] = bf.p[A][fi];
            v[sb] = aa ? vb[A][0][fi] : cell_vhat(g, prim, psi, alp, B, cs);
        }
        if (ba) {
            mc_face<double>(q[0], q[1], q[2], q[3], qBaL, qBaR);
            mc_face<double>(v[0], v[1], v[2], v[3], vbL, vbR);
        } else {
            qBaL = qBaR = q[0];
            vbL = vbR = v[0];
        }
    }
    // speeds: each direction takes the larger alpha sqrt(gamma^dd) of its two faces at
    // the edge (1 in an inactive direction)
    const long long i0 = lin(g, c[0], c[1], c[2]);
    const long long sA = aa ? g.st[A] : 0, sB = ba ? g.st[B] : 0;
    double ca = 1.0, cb = 1.0;
    if (alp || psi) {
        double cab[2];
        edge_speeds(g, psi, alp, i0, aa, ba, sA, sB, cab);
        ca = cab[0];
        cb = cab[1];
    }
    // step (iv), the upwind formula of App. A (sqrt(gamma_hat) = 1); with c+ = c- each
    // term (c v_R q_R + c v_L q_L - c^2 (q_R - q_L)) / 2c is
    // (v_R q_R + v_L q_L - c (q_R - q_L)) / 2
    Eh[i0] = -(vaR * qBbR + vaL * qBbL - ca * (qBbR - qBbL)) * 0.5 +
             (vbR * qBaR + vbL * qBaL - cb * (qBaR - qBaL)) * 0.5;
}

// ---------------------------------------------------------------------------
// update (Sec. 2.1 sources, Sec. 3.2 CT, Sec. 2.3 stage folds): item t = cell/face t
// ---------------------------------------------------------------------------

__device__ __forceinline__ void out_value(const UpdateArgs& a, int v, long long o, double L, bool has_r)
{
    if (a.mode == UPD_WRITE_L) {
        a.L[v][o] = L;
        return;
    }
    // base_k += dt (At[k][i] L + A[k][i] R), acc += dt (wt[i] L + w[i] R), with the
    // dt products formed on the host; q^n is read at stage 0 only
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

// the same for L = -S / (2 dx_0) without a stiff rate, stage folds only
__device__ __forceinline__ void out_scaled(const UpdateArgs& a, int v, long long o, double S)
{
    const double qn = a.stage == 0 ? a.qn[v][o] : 0.0;
    for (int k = a.stage + 1; k < a.s; k++) {
        const double prev = a.stage == 0 ? qn : a.base[k][v][o];
        a.base[k][v][o] = fma(a.cLS[k], S, prev);
    }
    const double nv = fma(a.cwLS, S, a.stage == 0 ? qn : a.acc[v][o]);
    if (a.stage == a.s - 1) a.qn[v][o] = nv;
    else a.acc[v][o] = nv;
}

// non-stiff sources of the 8 cell-centred variables at interior cell c (linear index
// o), in src (Sec. 2.1, beta = 0, K_ij = 0): the Gauss-law charge term of s_E (src[5..7])
// and, with a metric, s_S and s_tau (src[1..4]; src[0] stays unset).  bsrc: staggered face
// q_B, or cell q_B if CC.  qE: the solved q_E = psi^6 E^i of every interior cell, or NULL
// entries (then psi^6 E is formed here, as at cells beside a boundary, whose outer neighbour
// is the mapped cell's E with the metric stored in the ghost).
template <bool M, bool CC>
__device__ __forceinline__ void cell_sources(const Dims& g, const double* const* prim, const double* const* bsrc,
                                             const double* const* qE, const double* __restrict__ psi,
                                             const double* __restrict__ alp, const int* c, long long o, double* src)
{
    const double ps = psi ? psi[o] : 1.0;
    const double al = alp ? alp[o] : 1.0;
    const double p2 = ps * ps, p4 = p2 * p2, p6 = p4 * p2;
    double u[3];
#pragma unroll
    for (int i = 0; i < 3; i++) u[i] = prim[1 + i][o];
    const double u2 = fma(u[0], u[0], fma(u[1], u[1], u[2] * u[2]));
    const double xw = M ? fma(p4, u2, 1.0) : 1.0 + u2;
    const double iW = rsqrt_wide(xw);
    // Gauss law: sqrt(gamma) rho_e = div q_E by central differences
    double divqE = 0.0;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        if (!g.act[d]) continue;
        const bool edge = c[d] == g.ng[d] || c[d] == g.ng[d] + g.n[d] - 1;
        double qp, qm;
        if (M && qE && qE[d] && !edge) {
            qp = qE[d][chk(g, o + g.st[d])];
            qm = qE[d][chk(g, o - g.st[d])];
        } else {
            int cp[3] = {c[0], c[1], c[2]}, cm[3] = {c[0], c[1], c[2]};
            cp[d] += 1;
            cm[d] -= 1;
            qp = prim[5 + d][cell_at(g, cp)];
            qm = prim[5 + d][cell_at(g, cm)];
            if (psi) {
                double sp = psi[chk(g, o + g.st[d])], sm = psi[chk(g, o - g.st[d])];
                sp = sp * sp;
                sm = sm * sm;
                qp *= sp * sp * sp;
                qm *= sm * sm * sm;
            }
        }
        divqE += (qp - qm) * (0.5 * g.idx[d]);
    }
    // s_E (non-stiff part) = -alpha sqrt(gamma) rho_e v^i
    const double k = (M ? al * divqE : divqE) * iW;
#pragma unroll
    for (int i = 0; i < 3; i++) src[5 + i] = -k * u[i];
    if (psi || alp) {
        // s_S and s_tau for beta = 0, K_ij = 0 (Sec. 2.1) in the orthonormal frame:
        //   s_S_i = psi^6 [-(tau + D) d_i alpha + 2 alpha (d_i psi / psi)(rho h W^2 v^2 + 3p + U)]
        //   s_tau = -psi^4 S_hat_i d_i alpha
        // (the trace rho h W^2 v^2 + 3p + U is summed from its positive terms: as (tau + D) - rho h
        // + 4p it would lose the digits of p / rho in a cold gas, where it is the whole source of
        // a metric with psi alone)
        const double rho = prim[0][o], p = prim[4][o];
        const double ip4 = rcp_pos(p4);   // psi^-4; psi^-1 = psi^3 psi^-4
        double uh[3], Eh[3], Bh[3];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            uh[i] = p2 * u[i];
            Eh[i] = p2 * prim[5 + i][o];
            Bh[i] = (CC ? bsrc[i][o] : cell_qB_in(g, bsrc[i], i, c, o)) * ip4;   // psi^2 q_B / psi^6
        }
        const double rhoh = fma(g.gh, p, rho), W = xw * iW, hW = rhoh * W;
        const double U2 = fma(Eh[0], Eh[0], fma(Eh[1], Eh[1], fma(Eh[2], Eh[2], fma(Bh[0], Bh[0], fma(Bh[1], Bh[1], Bh[2] * Bh[2])))));
        const double tauD = fma(hW, W, fma(0.5, U2, -p));   // tau + D
        const double tr = fma(rhoh, p4 * u2, fma(3.0, p, 0.5 * U2));
        const double ktr = 2.0 * al * (ps * p2 * ip4) * tr;
        double s4 = 0.0;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            if (!g.act[i]) {
                src[1 + i] = 0.0;
                continue;
            }
            const int j = (i + 1) % 3, l = (i + 2) % 3;
            const double S = fma(hW, uh[i], fma(Eh[j], Bh[l], -(Eh[l] * Bh[j])));
            const double da = alp ? alp[chk(g, o + g.st[i])] - alp[chk(g, o - g.st[i])] : 0.0;
            const double dp = psi ? psi[chk(g, o + g.st[i])] - psi[chk(g, o - g.st[i])] : 0.0;
            const double h = 0.5 * g.idx[i];
            src[1 + i] = (p6 * h) * fma(ktr, dp, -tauD * da);
            s4 = fma(S, da * h, s4);
        }
        src[4] = -p4 * s4;
    }
}

// The same sources on the mixed-precision path, in FP32 from the stage's FP32
// primitives and cell q_B (the values its FP32 fluxes were built from).  The metric differences d_i alpha, d_i psi are
// taken in FP64 before rounding (a slowly varying alpha would otherwise lose digits to
// cancellation); the rest carries FP32 rounding, below the FP32 fluxes' own error.  src as
// cell_sources.
__device__ __forceinline__ void cell_sources_f32(const Dims& g, const float* const* p32,
                                                 const double* __restrict__ psi, const double* __restrict__ alp,
                                                 const int* c, long long o, float* src)
{
    const float ps = psi ? d2f_int(psi[o]) : 1.0f;
    const float al = alp ? d2f_int(alp[o]) : 1.0f;
    const float p2 = ps * ps, p4 = p2 * p2, p6 = p4 * p2;
    float u[3];
#pragma unroll
    for (int i = 0; i < 3; i++) u[i] = p32[1 + i][o];
    const float xw = 1.0f + p4 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    const float iW = rsqrtf(xw);
    const float W = xw * iW;
    float divqE = 0.0f;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        if (!g.act[d]) continue;
        int cp[3] = {c[0], c[1], c[2]}, cm[3] = {c[0], c[1], c[2]};
        cp[d] += 1;
        cm[d] -= 1;
        float sp = psi ? d2f_int(psi[chk(g, o + g.st[d])]) : 1.0f, sm = psi ? d2f_int(psi[chk(g, o - g.st[d])]) : 1.0f;
        sp = sp * sp;
        sm = sm * sm;
        const float qp = sp * sp * sp * p32[5 + d][cell_at(g, cp)];
        const float qm = sm * sm * sm * p32[5 + d][cell_at(g, cm)];
        divqE += (qp - qm) * (0.5f * d2f_int(g.idx[d]));
    }
#pragma unroll
    for (int i = 0; i < 3; i++) src[5 + i] = -(al * divqE * (u[i] * iW));
    if (psi || alp) {
        const float rho = p32[0][o], p = p32[4][o];
        const float ip4 = 1.0f / p4, ips = ps * p2 * ip4;   // psi^-4, psi^-1
        float uh[3], Eh[3], Bh[3];
#pragma unroll
        for (int i = 0; i < 3; i++) {
            uh[i] = p2 * u[i];
            Eh[i] = p2 * p32[5 + i][o];
            Bh[i] = p32[8 + i][o] * ip4;   // psi^2 q_B / psi^6
        }
        const float rhoh = rho + d2f_int(g.gh) * p;
        const float U = 0.5f * (Eh[0] * Eh[0] + Eh[1] * Eh[1] + Eh[2] * Eh[2] + Bh[0] * Bh[0] + Bh[1] * Bh[1] +
                                Bh[2] * Bh[2]);
        const float tauD = rhoh * W * W - p + U;   // tau + D
        float S[3];
        S[0] = rhoh * W * uh[0] + (Eh[1] * Bh[2] - Eh[2] * Bh[1]);
        S[1] = rhoh * W * uh[1] + (Eh[2] * Bh[0] - Eh[0] * Bh[2]);
        S[2] = rhoh * W * uh[2] + (Eh[0] * Bh[1] - Eh[1] * Bh[0]);
        const float tr = rhoh * (uh[0] * uh[0] + uh[1] * uh[1] + uh[2] * uh[2]) + 3.0f * p + U;
        float s4 = 0.0f;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            if (!g.act[i]) {
                src[1 + i] = 0.0f;
                continue;
            }
            const long long op = chk(g, o + g.st[i]), om = chk(g, o - g.st[i]);
            const float hi = 0.5f * d2f_int(g.idx[i]);
            const float dal = alp ? d2f_int(alp[op] - alp[om]) * hi : 0.0f;
            const float dps = psi ? d2f_int(psi[op] - psi[om]) * hi : 0.0f;
            src[1 + i] = p6 * (-tauD * dal + 2.0f * al * (dps * ips) * tr);
            s4 += S[i] * dal;
        }
        src[4] = -(p4 * s4);
    }
}

template <bool M, bool F32 = false, bool ALL = false>
__device__ __forceinline__ void update_item(const Dims& g, const UpdateArgs& a, long long t)
{
    // flat metric: alpha = psi = 1 known at compile time
    const double* __restrict__ psi = M ? a.psi : nullptr;
    const double* __restrict__ alp = M ? a.alp : nullptr;
    // cells and their upper faces: n[d] + 1 along an active d
    int c[3];
    box_coords(t, g.dvp[0], g.dvp[1], c);
#pragma unroll
    for (int d = 0; d < 3; d++) c[d] += g.ng[d];
    bool interior = true;
#pragma unroll
    for (int d = 0; d < 3; d++)
        if (c[d] >= g.ng[d] + g.n[d]) interior = false;
    const long long o = lin(g, c[0], c[1], c[2]);
    if (interior) {
        // which variables have a source: E, and with a metric S and tau
        auto sourced = [](int v) { return v >= 5 || (M && v >= 1); };
        if (F32) {
            // The fluxes are FP32 arrays (mixed precision).  Each difference of two FP32 values
            // is exact as a double-word, and the divergence sum_d (F[o + e_d] - F[o]) / (2 dx_d)
            // is formed in double-word arithmetic on the FP32 pipe (about 2^-46 of its terms,
            // far below the FP32 fluxes' own error) and widened by one FP64 add, in place of two
            // FP64 instructions per flux.
            float src[8];
            if (!ALL) cell_sources_f32(g, a.p32, psi, alp, c, o, src);
            auto divergence = [&](int v) {
                dw acc = dw_make(0.0f);
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    if (!g.act[d]) continue;
                    const dw h = {g.hix[d][0], g.hix[d][1]};   // F holds twice the flux
                    const float* __restrict__ Fv = reinterpret_cast<const float*>(a.F[d][v]);
                    const dw term = dw_mul(two_sum(Fv[chk(g, o + g.st[d])], -Fv[o]), h);
                    acc = d == 0 ? term : dw_add(acc, term);   // (direction 0 is always active)
                }
                return acc;
            };
            // ALL: every variable's flux loads before the first store, which the compiler does
            // not move loads across
            dw all[8];
#pragma unroll
            for (int v = 0; v < 8; v++)
                if (ALL) all[v] = divergence(v);
            if (ALL) cell_sources_f32(g, a.p32, psi, alp, c, o, src);
#pragma unroll
            for (int v = 0; v < 8; v++) {
                double L = -dw_to_double(ALL ? all[v] : divergence(v));
                if (sourced(v)) L += f2d_int(src[v]);
                out_value(a, v, o, L, v >= 5);
            }
        } else {
            // F holds twice the flux: L = -(dF_0 + (dx_0/dx_1) dF_1 + ...) / (2 dx_0) + source.
            // Flat: the flux loads of a direction are issued together (the kernel waits on
            // memory: 512^2 61.5 -> 55.7 us); with a metric one variable at a time (its
            // sources hold the registers: 128^3 866 -> 748 us).
            double src[8];
            auto put = [&](int v, double S) {
                if (sourced(v) || a.mode == UPD_WRITE_L)
                    out_value(a, v, o, fma(-0.5 * g.idx[0], S, sourced(v) ? src[v] : 0.0), v >= 5);
                else out_scaled(a, v, o, S);   // the factor folded into the stage weights
            };
            if (M) {
                cell_sources<M, false>(g, a.prim, a.bf, a.qE, psi, alp, c, o, src);
#pragma unroll
                for (int v = 0; v < 8; v++) {
                    double S = 0.0;
#pragma unroll
                    for (int d = 0; d < 3; d++) {
                        if (!g.act[d]) continue;
                        const double* __restrict__ Fv = a.F[d][v];
                        const double df = Fv[chk(g, o + g.st[d])] - Fv[o];
                        S = d == 0 ? df : fma(df, g.rdx[d], S);
                    }
                    put(v, S);
                }
            } else {
                double S[8];
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    if (!g.act[d]) continue;
                    const long long o1 = chk(g, o + g.st[d]);
#pragma unroll
                    for (int v = 0; v < 8; v++) {
                        const double* __restrict__ Fv = a.F[d][v];
                        const double df = Fv[o1] - Fv[o];
                        S[v] = d == 0 ? df : fma(df, g.rdx[d], S[v]);
                    }
                }
                cell_sources<M, false>(g, a.prim, a.bf, a.qE, psi, alp, c, o, src);
#pragma unroll
                for (int v = 0; v < 8; v++) put(v, S[v]);
            }
        }
    }
    // CT: d q_B^fa / dt = -d_fb hat{E}_fc + d_fc hat{E}_fb  (fa, fb, fc cyclic)
#pragma unroll
    for (int fa = 0; fa < 3; fa++) {
        const int fb = (fa + 1) % 3, fc = (fa + 2) % 3;
        bool ok = true;
#pragma unroll
        for (int d = 0; d < 3; d++) {
            int hi = g.ng[d] + g.n[d] - 1;
            if (d == fa && g.act[d] && g.bc[d] != BC_PERIODIC) hi += 1;
            if (c[d] > hi) ok = false;
        }
        if (!ok) continue;
        double r = 0.0;
        const double* __restrict__ Ec = a.Eh[fc];
        const double* __restrict__ Eb = a.Eh[fb];
        if (g.act[fb]) r -= (Ec[chk(g, o + g.st[fb])] - Ec[o]) * g.idx[fb];
        if (g.act[fc]) r += (Eb[chk(g, o + g.st[fc])] - Eb[o]) * g.idx[fc];
        out_value(a, 8 + fa, o, r, false);
    }
}

// edges of direction C (one per thread when A or B is inactive)
inline long long emf_work(const Dims& g, int c)
{
    long long work = 1;
    for (int d = 0; d < 3; d++) work *= (d == c) ? g.n[d] : (g.act[d] ? g.n[d] + 1 : 1);
    return work;
}

}  // namespace grmhd
