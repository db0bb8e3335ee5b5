"""The per-cell device code (csrc/*.cuh) compiled as plain C++ (device_on_host.h) and run on
the CPU at inputs where a rule inside it can go wrong."""
import math
import shutil
import subprocess
from decimal import Decimal, getcontext
from fractions import Fraction as Fr
from pathlib import Path

import numpy as np
import pytest

ROOT = Path(__file__).resolve().parents[1]
CUDA = Path(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc").resolve().parents[1] / "include"

pytestmark = pytest.mark.skipif(shutil.which("g++") is None or not (CUDA / "cuda_runtime.h").exists(),
                                reason="no g++ or CUDA headers")


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """The rows (lists of floats) through the program `src`, a list of floats back for each."""
    built = {}

    def call(src, rows, *flags):
        if src not in built:
            d = tmp_path_factory.mktemp("device")
            (d / "t.cpp").write_text('#include "device_on_host.h"\n' + src)
            inc = [ROOT / "tests", CUDA, ROOT / "paper_2110_03732_gb300" / "csrc", ROOT / "include"]
            subprocess.run(["g++", "-O0", "-std=c++17", "-ffp-contract=off", "-pthread", "-ffunction-sections",
                            "-Wl,--gc-sections", *flags, *(f"-I{i}" for i in inc), str(d / "t.cpp"),
                            "-o", str(d / "t")], check=True)
            built[src] = d / "t"
        text = "\n".join(" ".join(float(x).hex() for x in r) for r in rows) + "\n"
        out = subprocess.run([str(built[src])], input=text, capture_output=True, text=True, check=True).stdout
        return [[float.fromhex(x) for x in ln.split()] for ln in out.splitlines()]

    return call


GRID = r"""
#include <cstdio>
#include "grmhd_device.cuh"
#include "items.cuh"
using namespace grmhd;
// a 1-D grid of four cells
Dims grid4()
{
    Dims g = {};
    g.n[0] = 4; g.n[1] = g.n[2] = 1;
    g.ng[0] = 2; g.N[0] = 8; g.N[1] = g.N[2] = 1;
    g.act[0] = 1;
    g.st[0] = 1; g.st[1] = g.st[2] = 8;
    g.idx[0] = 4.0;
    g.gh = 4.0; g.igh = 0.25;
    g.ncell = 8;
    set_divisors(g);
    return g;
}
"""

# a state in a flat cell and its solve from another start: prints the failures, rho, u and p,
# how often the general solve and the double-word corrections were entered (with
# -finstrument-functions), and the FP32 copy
IMPLICIT = GRID + r"""
static int general, refine;
#define HOOK extern "C" __attribute__((no_instrument_function)) void
HOOK __cyg_profile_func_exit(void*, void*) {}
HOOK __cyg_profile_func_enter(void* f, void*)
{
    general += f == (void*)implicit_general<false, false, ACC, false>;
    refine += f == (void*)newton_refine_dw<ACC>;
}
int main() {
    double s, r, a_dt, us, u0;   // density scale, field scale, a_ii dt, velocity scale, start
    while (std::scanf("%la %la %la %la %la", &s, &r, &a_dt, &us, &u0) == 5) {
        const Dims g = grid4();
        const double rho = 1.3 * s, p = 0.7 * s, u[3] = {0.4 * us, -0.6 * us, 0.3 * us}, E[3] = {0.5 * r, 0.2 * r, -0.3 * r},
                     B[3] = {0.6 * r, -0.8 * r, 0.5 * r};
        const double W = std::sqrt(1 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]), hW = (rho + 4.0 * p) * W;
        double q[8], U = 0;
        for (int i = 0; i < 3; i++) U += 0.5 * (E[i] * E[i] + B[i] * B[i]);
        q[0] = rho * W;
        for (int i = 0; i < 3; i++) {
            const int j = (i + 1) % 3, k = (i + 2) % 3;
            q[1 + i] = hW * u[i] + E[j] * B[k] - E[k] * B[j];
            q[5 + i] = E[i];
        }
        q[4] = hW * W - p + U - q[0];
        double A[30][8];
        ImpArgs a = {};
        for (int v = 0; v < 8; v++) {
            for (int c = 0; c < 8; c++) A[v][c] = q[v];
            a.qb.p[v] = A[v];
            a.prim.p[v] = A[11 + v];
        }
        const double start[8] = {s, u0, u0, u0, s, 0, 0, 0};
        for (int c = 0; c < 8; c++)
            for (int v = 0; v < 8; v++) A[11 + v][c] = start[v];
        for (int d = 0; d < 3; d++) {
            for (int c = 0; c < 8; c++) A[8 + d][c] = B[d];
            a.bf.p[d] = A[8 + d];
            a.R.p[d] = A[19 + d];
            a.qE_out.p[d] = A[22 + d];
        }
        unsigned long long nfail = 0;
        a.eta_u = 0.01;
        a.a_dt = a_dt;
        a.ia_dt = a_dt > 0 ? 1 / a_dt : 0;
        a.stiff = a_dt > 0;
        a.ighf = 0.25f;
        a.kmax = 100;
        a.tol = 1e-13;
        a.tolf = 1e-13f;
        a.nfail = &nfail;
        static float f32[11][8];
        for (int v = 0; v < 11; v++) {
            a.p32.p[v] = f32[v];
            f32[v][3] = -1.0f;
        }
        if (ACC) {
            a.tol = 1e-10;
            a.tolf = 1e-10f;
        }
        general = refine = 0;
        implicit_item<false, false, ACC>(g, a, 1);
        std::printf("%a %a %a %a %a %a %a %a ", (double)nfail, A[11][3] / s, A[12][3], A[13][3], A[14][3], A[15][3] / s,
                    (double)general, (double)refine);
        for (int v = 0; v < 11; v++) std::printf("%a ", (double)f32[v][3]);
        std::printf("\n");
    }
}
"""


def implicit(run, rows, acc=False):
    return run(IMPLICIT.replace("ACC", str(acc).lower()), rows, "-finstrument-functions")


@pytest.mark.parametrize("a_dt", [0.0, 0.05])
def test_implicit_solve_at_any_scale(run, a_dt):
    """The equations of the implicit solve do not change when densities are multiplied by s and
    fields by its root: the velocity and the scaled density and pressure stay the same, also where
    the momentum leaves the range of FP32.  1e-11: the 1e-13 of the residual test on both
    sides, and the condition of this state (below 10)."""
    r = [2.0 ** k for k in (0, -40, 40, 64, 70, 100)]
    rows = implicit(run, [[x * x, x, a_dt, 1.0, 0.1] for x in r])
    assert all(row[0] == 0 for row in rows)
    if a_dt == 0.0:   # E held fixed: the state itself is the root
        assert rows[0][1:6] == pytest.approx([1.3, 0.4, -0.6, 0.3, 0.7], rel=1e-11)
    for row in rows[1:]:
        assert row[1:6] == pytest.approx(rows[0][1:6], rel=1e-11)


@pytest.mark.parametrize("acc", [False, True])
@pytest.mark.parametrize("a_dt", [0.0, 0.05])
def test_cell_at_rest_takes_the_direct_path(run, a_dt, acc):
    """A cell without momentum has the momentum scale zero: its start u = 0 solves it exactly, and
    the direct path accepts that."""
    for row in implicit(run, [[s, 0.0, a_dt, 0.0, 0.0] for s in (1.0, 1e-12, 1e6)], acc):
        assert row[:1] + row[2:5] == [0.0] * 4 and [row[1], row[5]] == pytest.approx([1.3, 0.7], rel=1e-14)
        assert row[6] == 0


@pytest.mark.parametrize("a_dt", [0.0, 0.05])
@pytest.mark.parametrize("r", [0.0, 1e-6])
def test_slow_cell_takes_the_direct_path(run, a_dt, r):
    """The residual is measured by the cell's own momentum, so a start a few times off is corrected
    to it on the direct path however slow the cell is.  (1e-12: ten times the tolerance; with
    fields the momentum is their E x B, and that relative to it.)"""
    for row in implicit(run, [[1.0, r * us, a_dt, us, 3 * us] for us in (1e-3, 1e-6, 1e-10, 1e-16, 1e-22)]):
        assert row[0] == 0 and row[6] == 0
        if a_dt == 0.0 or r == 0.0:
            assert row[3] / row[2] == pytest.approx(-1.5, rel=1e-12) and row[4] / row[2] == pytest.approx(0.75, rel=1e-12)


@pytest.mark.parametrize("us,u0", [(1.0, 0.1), (0.0, 0.0), (20.0, 0.0)])
def test_only_the_mixed_solve_writes_the_fp32_copy(run, us, u0):
    """On the direct path, at rest and through the general solve: the rounded primitives and field
    in mixed precision, nothing in FP64 (which has no such copy)."""
    r = 0.0 if us == 0.0 else 1.0
    assert implicit(run, [[1.0, r, 0.0, us, u0]])[0][8:] == [-1.0] * 11
    row = implicit(run, [[1.0, r, 0.0, us, u0]], acc=True)[0]
    want = row[1:6] + [0.5 * r, 0.2 * r, -0.3 * r, 0.6 * r, -0.8 * r, 0.5 * r]
    assert row[8:] == [float(np.float32(x)) for x in want]


@pytest.mark.parametrize("acc", [False, True])
@pytest.mark.parametrize("a_dt", [0.0, 0.05])
def test_refused_cell_goes_on_from_the_corrections(run, a_dt, acc):
    """A cell whose double-word corrections do not reach the root goes on in FP64 from where they
    ended: they run once.  (The result: to the residual's tolerance times the condition of w_t in
    the velocity at u = 20, W^2 = 400.)"""
    rows = implicit(run, [[1.0, 1.0, a_dt, 20.0, x] for x in (0.0, 0.01)], acc)
    near = implicit(run, [[1.0, 1.0, a_dt, 20.0, rows[0][2]]], acc)[0]
    for row in rows:
        assert row[0] == 0 and row[1:6] == pytest.approx(near[1:6], rel=4e-8 if acc else 4e-11)
    assert any(row[6] == 1 for row in rows)
    assert all(row[7] == 1 for row in rows)


# which kernel the implicit solve launches for (psi set, xi, mixed precision, cell-centred field)
KERNELS = r"""
#include <cuda_runtime.h>
static const void* fn;
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* k, void**)
{
    fn = k;
    return cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
#define asm
#define volatile(...)   // (griddepcontrol)
""" + GRID + r"""
#include "implicit.cu"
namespace grmhd { thread_local bool launch_overlap; }
int main() {
    double m, xi, acc, cc;
    while (std::scanf("%la %la %la %la", &m, &xi, &acc, &cc) == 4) {
        const Dims g = grid4();
        ImpArgs a = {};
        double psi;
        a.psi = m ? &psi : nullptr;
        a.xi = xi;
        a.dwacc = (int)acc;
        if (cc) launch_implicit_cc(g, a, 152, nullptr);
        else launch_implicit(g, a, 152, nullptr);
        const void* const all[] = {(void*)k_implicit_dynamo<false, false, false>, (void*)k_implicit_dynamo<true, false, false>,
                                   (void*)k_implicit_dynamo<false, false, true>, (void*)k_implicit_dynamo<true, false, true>,
                                   (void*)k_implicit_dynamo<false, true, false>, (void*)k_implicit_dynamo<true, true, false>};
        std::printf("%d\n", (int)(std::find(all, all + 6, fn) - all) + 1);
    }
}
"""


def test_dynamo_form_has_its_own_kernel(run):
    """xi != 0 launches the kernel with the general solve inline, of the same variant; xi = 0 does not."""
    rows = [[m, xi, acc, cc] for xi in (0.3, -1e-300, 0.0) for cc in (0, 1) for acc in (0, 1) for m in (0, 1)
            if not (cc and acc)]
    got = [r[0] for r in run(KERNELS, rows)]
    assert got == [7 if xi == 0.0 else 1 + m + 2 * acc + 4 * cc for m, xi, acc, cc in rows]


# the sources of a cell on a metric with psi alone
SOURCES = GRID + r"""
int main() {
    double rho, p, f;   // density, pressure, size of u, E and B
    while (std::scanf("%la %la %la", &rho, &p, &f) == 3) {
        const Dims g = grid4();
        double A[11][8], psi[8], src[8];
        const double st[11] = {rho, f, -2 * f, f, p, 2 * f, f, -f, f, f, 2 * f};
        const double *prim[8], *bf[3];
        for (int c = 0; c < 8; c++) {
            for (int v = 0; v < 11; v++) A[v][c] = st[v];
            psi[c] = 1.0 + 0.125 * c;
        }
        for (int v = 0; v < 8; v++) prim[v] = A[v];
        for (int d = 0; d < 3; d++) bf[d] = A[8 + d];
        const int c[3] = {4, 0, 0};
        cell_sources<true, false>(g, prim, bf, nullptr, psi, nullptr, c, 4, src);
        std::printf("%a\n", src[1]);
    }
}
"""


def test_momentum_source_of_a_cold_gas(run):
    """s_S = psi^6 2 alpha (d psi / psi) (rho h W^2 v^2 + 3 p + U) (Sec. 2.1) where the pressure and
    the fields are far below the rest mass: a sum of positive terms, so 1e-14 (thirty roundings of
    2^-53, and the reciprocal of psi^4 to an ulp or so) holds whatever their size."""
    rows = [[rho, rho * 10.0 ** -k, m] for rho in (1.0, 1e-13) for k in (1, 5, 8, 11) for m in (0.0, 1e-9, 0.5)]
    for (rho, p, f), (got,) in zip(rows, run(SOURCES, rows)):
        rho, p, f, psi = Fr(rho), Fr(p), Fr(f), Fr(3, 2)
        u2, U = psi ** 4 * 6 * f * f, (psi ** 4 * 6 * f * f + 6 * f * f / psi ** 8) / 2
        want = psi ** 6 * 2 * (Fr(1, 4) * 2 / psi) * ((rho + 4 * p) * u2 + 3 * p + U)
        assert abs(Fr(got) - want) <= want / 10 ** 14


# the Lorentz factor of an HLL half; the transport velocity u^t / W of a uniform state at a face;
# the charge-current source -div q_E u^t / W
LORENTZ = GRID + r"""
int main() {
    double u;
    while (std::scanf("%la", &u) == 1) {
        const Dims g = grid4();
        const double st[8] = {1, u, 2 * u, 2 * u, 1, 0.1, 0.2, 0.3}, Bt[2] = {0.5, 0.25};
        double gh[8], W, A[11][8], F[8][8], vb[2][8], src[8];
        const double *prim[8], *bf[3];
        double *Fp[8], *vbar[2] = {vb[0], vb[1]};
        hll_half64<1>(st, Bt, 0.5, 0.125, 4.0, gh, W);
        for (int c = 0; c < 8; c++)
            for (int v = 0; v < 11; v++) A[v][c] = v < 8 ? st[v] : 0.5;
        for (int v = 0; v < 8; v++) {
            prim[v] = A[v];
            Fp[v] = F[v];
        }
        for (int d = 0; d < 3; d++) bf[d] = A[8 + d];
        static double sm[Flux64<false, false>::SM];
        flux64_item<false, false, false>(g, 0, prim, bf, nullptr, nullptr, nullptr, Fp, vbar, nullptr, sm, 1);
        for (int c = 0; c < 8; c++) A[5][c] = c;   // d_x E^x = 4
        const int c[3] = {4, 0, 0};
        cell_sources<false, false>(g, prim, bf, nullptr, nullptr, nullptr, c, 4, src);
        std::printf("%a %a %a\n", W, vb[0][3], src[6]);
    }
}
"""


def test_lorentz_factor_at_any_velocity(run):
    """W = sqrt(1 + u^2) and u^t / W over the whole range of FP64 squares, also where 1 + u^2 or W
    leaves the range of the FP32 estimates (u = 6e18 and 3e37): two ulp each."""
    us = [0.0, 1e-3, 1.0, 1e9, 4e18, 8e18, 1e25, 2e37, 5e37, 1e100, 1e150]
    getcontext().prec = 40
    for u, (W, v, s) in zip(us, run(LORENTZ, [[u] for u in us])):
        want = (1 + 9 * Decimal(u) ** 2).sqrt()
        tol = Decimal(2) ** -51
        assert abs(Decimal(W) - want) <= tol * want
        assert abs(Decimal(v) - 2 * Decimal(u) / want) <= tol
        assert abs(Decimal(s) + 8 * Decimal(u) / want) <= 4 * tol
    bad = run(LORENTZ, [[float("nan")], [1e200]])
    assert all(math.isnan(r[0]) for r in bad)   # (the square of 1e200 is infinite)


# The one-warp coarse solve of the multigrid cleaning with every lane on its own copy of the
# vectors: what a lane writes reaches the others at a warp barrier only, which is all that CUDA
# promises (shuffles order no memory).
COARSE = r"""
#include <atomic>
#include <thread>
#include <vector>
struct Meet {   // a barrier of 32 threads
    std::atomic<int> n{0}, round{0};
    void wait()
    {
        const int r = round;
        if (++n == 32) {
            n = 0;
            round++;
        } else
            while (round == r) std::this_thread::yield();
    }
} meet;
constexpr int kMax = 64;
double vec[32][5][kMax], slot[32];   // per lane: phi, res, p, q, rhs
int cells;
inline void __syncthreads() {}
inline void __syncwarp()
{
    meet.wait();
    const int l = threadIdx.x;
    for (int v = 0; v < 4; v++)
        for (int t = l; t < cells; t += 32)
            for (int o = 0; o < 32; o++) vec[o][v][t] = vec[l][v][t];
    meet.wait();
}
inline double __shfl_xor_sync(unsigned, double v, int o)
{
    slot[threadIdx.x] = v;
    meet.wait();
    const double r = slot[threadIdx.x ^ o];
    meet.wait();
    return r;
}
inline double __shfl_down_sync(unsigned, double v, int) { return v; }
#include <cstdio>
#define __shared__
#define asm
#define volatile(...)   // (griddepcontrol)
#include "elliptic.cu"
namespace grmhd { namespace { double tail_sm[1]; } }
using namespace grmhd;
int main() {
    double n0, n1, bc;
    while (std::scanf("%la %la %la", &n0, &n1, &bc) == 3) {
        MgLevel L = {};
        const int b = bc ? BC_OUTFLOW : BC_PERIODIC;
        MgArgs m = {{b, b, b}, {1, 1, 0}};
        L.n[0] = (int)n0; L.n[1] = (int)n1; L.n[2] = 1;
        L.ih2[0] = 4.0; L.ih2[1] = 1.0;
        L.dfull = 10.0;
        L.f0 = make_fastdiv(L.n[0]);
        L.f1 = make_fastdiv(L.n[1]);
        L.cells = cells = L.n[0] * L.n[1];
        for (int l = 0; l < 32; l++)
            for (int t = 0; t < cells; t++) {
                for (int v = 0; v < 4; v++) vec[l][v][t] = NAN;
                vec[l][4][t] = (t * 37 % 19) - 9.0;
            }
        std::vector<std::thread> lanes;
        for (int l = 0; l < 32; l++)
            lanes.emplace_back([=] {
                threadIdx.x = l;
                MgLevel M = L;
                double sh[33];
                M.phi = vec[l][0];
                M.rhs = vec[l][4];
                mg_cg_run<true>(M, m, vec[l][1], vec[l][2], vec[l][3], 2 * cells + 20, sh);
            });
        for (auto& x : lanes) x.join();
        for (int t = 0; t < cells; t++) std::printf("%a ", vec[t % 32][0][t]);
        std::printf("\n");
    }
}
"""


@pytest.mark.parametrize("n0,n1", [(4, 4), (5, 5), (7, 7), (8, 8), (2, 31)])
@pytest.mark.parametrize("bc", ["periodic", "outflow"])
def test_one_warp_coarse_solve(run, n0, n1, bc):
    """The lanes' result solves the 5-point problem.  Conjugate gradients stop at 1e-15 of the
    right-hand side (values up to 9); the operator's norm is below 20: residual <= 1e-12."""
    phi = np.array(run(COARSE, [[n0, n1, bc == "outflow"]])[0]).reshape(n1, n0)
    rhs = ((np.arange(n0 * n1) * 37 % 19) - 9.0).reshape(n1, n0)
    mode = "wrap" if bc == "periodic" else "edge"
    e = np.pad(phi, 1, mode=mode)
    lap = 4.0 * (e[1:-1, 2:] - 2 * phi + e[1:-1, :-2]) + (e[2:, 1:-1] - 2 * phi + e[:-2, 1:-1])
    assert np.abs(lap - (rhs - rhs.mean())).max() <= 1e-12


# mg_clean with the CUDA runtime's launch call replaced: each launch's grid, block and shared bytes
# are printed, and launch `bad` (counted from 0; -1: none) is refused
LAUNCHES = r"""
#include <cstdio>
#include <cuda_runtime.h>
static int launched, bad;
static const void* fn[4096];
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* k, void**)
{
    if (launched == bad) return launched++, cudaErrorInvalidValue;
    fn[launched++] = k;
    for (size_t v : {(size_t)c->gridDim.x, (size_t)c->gridDim.y, (size_t)c->gridDim.z, (size_t)c->blockDim.x,
                     c->dynamicSmemBytes})
        std::printf("%a ", (double)v);
    return cudaSuccess;
}
inline void __syncthreads() {}
inline void __syncwarp() {}
inline double __shfl_xor_sync(unsigned, double v, int) { return v; }
inline double __shfl_down_sync(unsigned, double v, int) { return v; }
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
#undef __shared__
#define __shared__
#define asm
#define volatile(...)   // (griddepcontrol)
#include "elliptic.cu"
namespace grmhd { thread_local bool launch_overlap; namespace { double tail_sm[1]; } }
using namespace grmhd;
int main() {
    double n[3], b;
    while (std::scanf("%la %la %la %la", n, n + 1, n + 2, &b) == 4) {
        Dims g = {};
        for (int d = 0; d < 3; d++) {
            g.n[d] = (int)n[d];
            g.act[d] = n[d] > 1;
            g.idx[d] = g.act[d];
        }
        set_divisors(g);
        launched = 0;
        bad = (int)b;
        MgPlan plan;
        double *bq[3] = {}, scratch[1];
        if (mg_plan(g, &plan) != 0) return 1;
        long long nl = 0;
        const cudaError_t e = mg_clean(g, plan, scratch, scratch, scratch, bq, false, 2, 152, nullptr, &nl);
        std::printf("%a %a %a\n", (double)e, (double)launched, (double)(fn[launched - 1] == (const void*)k_mg_correct));
    }
}
"""


def launches(run, n, bad=-1):
    r = [int(x) for x in run(LAUNCHES, [[*n, *[1] * (3 - len(n)), bad]])[0]]
    return [r[i:i + 5] for i in range(0, len(r) - 3, 5)], r[-3:]


@pytest.mark.parametrize("n", [(35, 35), (34, 36), (70, 70), (560, 560), (1120, 1120), (36, 34), (1223,), (9784,),
                               (17, 9, 8), (512, 512), (48, 48, 48)])
def test_cleaning_launches_fit_a_block(run, n):
    """Every launch's shared memory fits the 48 KB that a block has without opting in: the tail
    kernel's dynamic bytes with its static block sums (33 doubles, to the next 16 bytes)."""
    ls, (err, _, last) = launches(run, n)
    assert err == 0 and last == 1
    assert all(dyn + (33 * 8 + 8 if block == 1024 else 0) <= 48 * 1024 for *_, block, dyn in ls)


def test_cleaning_stops_at_a_refused_launch(run):
    """A refused launch ends the cleaning with its error: the field is not corrected by a
    potential that was not solved for."""
    total = len(launches(run, (96, 64))[0])
    for bad in range(total):
        _, (err, launched, last) = launches(run, (96, 64), bad)
        assert err == 1 and launched == bad + 1 and last == 0
