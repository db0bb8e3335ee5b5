"""Performance cases of the resistive-MHD solver: what a user's program has it do.

Every case is one call of a public entry point on a state that lives on the GPU: a
time step of a single problem (``Solver.step``), of many problems together
(``Batch.step``), or an elliptic cleaning (``Solver.clean_divb``).  The problems are the
ones of ``paper_2110_03732_gb300.problems`` (shock tube, Orszag-Tang vortex, magnetised
star, boxes of uneven sides), made on the GPU with seeded phases, resistivities and
perturbations, so that every component of every field is in play.

A state is stepped on from pass to pass, as a run does, and starts over from its
initial data after the run's usual number of steps.

``exact`` restates one step in plain torch, in 64 bits, from the paper's formulas.
"""
from __future__ import annotations

import math

import torch

DEVICE = "cuda"


def listed():
    return [
        # a 1-D run of the paper's Riemann problem: 400 cells, where launches and latency count
        dict(name="tube_400_fp64", kind="tube", n=400, precision="fp64", rec="mc"),
        # a served tube (they come with up to 4096 cells, in mixed precision), ragged
        dict(name="tube_2999_mixed", kind="tube", n=2999, precision="mixed", rec="mc"),
        # a small vortex, as in the batches and convergence runs
        dict(name="vortex_96_fp64", kind="vortex", n=96, precision="fp64", rec="mc", divb="ct"),
        # the headline workload and its mixed-precision form
        dict(name="vortex_512_fp64", kind="vortex", n=512, precision="fp64", rec="mc", divb="ct"),
        dict(name="vortex_512_mixed", kind="vortex", n=512, precision="mixed", rec="mc", divb="ct"),
        # the other reconstruction, at an odd side
        dict(name="vortex_301_ppm", kind="vortex", n=301, precision="fp64", rec="ppm", divb="ct"),
        # the other divergence control (cell-centred field with hyperbolic cleaning)
        dict(name="vortex_384_glm", kind="vortex", n=384, precision="fp64", rec="mc", divb="glm"),
        # the 3-D star on its curved metric: a served size, and the largest run
        dict(name="star_96_mixed", kind="star", n=96, precision="mixed", rec="mc"),
        dict(name="star_128_fp64", kind="star", n=128, precision="fp64", rec="mc"),
        dict(name="star_256_mixed", kind="star", n=256, precision="mixed", rec="mc"),
        # many vortices of uneven sides and resistivities advanced together
        dict(name="batch_24_mixed", kind="batch", boxes=24, lo=64, hi=400, mix=1, precision="mixed", rec="mc"),
        # elliptic cleaning of the staggered field of a 512^2 grid
        dict(name="clean_512", kind="clean", n=512, cycles=4, precision="fp64", rec="mc", divb="ct"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["tube", "tube", "vortex", "vortex", "vortex", "star", "star", "batch", "clean"])
    precision = rng.choice(["fp64", "mixed"])
    if kind == "tube":
        return dict(kind=kind, n=_log_int(rng, 200, 4096), precision=precision, rec="mc")
    if kind == "vortex":
        divb = rng.choice(["ct", "ct", "glm"])
        return dict(kind=kind, n=_log_int(rng, 48, 640), precision="fp64" if divb == "glm" else precision,
                    rec=rng.choice(["mc", "mc", "ppm"]), divb=divb)
    if kind == "star":
        return dict(kind=kind, n=_log_int(rng, 48, 160), precision=precision, rec="mc")
    if kind == "batch":
        lo = _log_int(rng, 48, 128)
        return dict(kind=kind, boxes=rng.randint(2, 32), lo=lo, hi=lo * rng.randint(2, 3), mix=rng.randint(0, 999),
                    precision=precision, rec="mc")
    return dict(kind=kind, n=16 * _log_int(rng, 4, 40), cycles=rng.randint(1, 6), precision="fp64", rec="mc", divb="ct")


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

class _Problem:
    """One problem's grid, parameters and initial data (padded tensors on the GPU)."""

    alpha = psi = eta = A = bface = phi = None
    eta_u = rho_atm = p_atm = kappa = 0.0
    cfl = 0.4
    divb = "ct"

    def axes(self, ndim, n, lo, hi, bc, gamma):
        self.ndim, self.bc, self.gamma = ndim, bc, gamma
        self.n = [n if d < ndim else 1 for d in range(3)]
        self.ng = [2 if d < ndim else 0 for d in range(3)]
        self.lo = [lo if d < ndim else 0.0 for d in range(3)]
        self.hi = [hi if d < ndim else 1.0 for d in range(3)]
        self.dx = [(self.hi[d] - self.lo[d]) / self.n[d] for d in range(3)]
        i = [torch.arange(self.n[d] + 2 * self.ng[d], dtype=torch.float64, device=DEVICE) for d in range(3)]
        self.face = [self.lo[d] + (i[d] - self.ng[d]) * self.dx[d] for d in range(3)]
        self.cent = [self.face[d] + 0.5 * self.dx[d] for d in range(3)]

    def mesh(self, on=()):
        """x, y, z on cells, or on the lower faces of the directions in `on`."""
        c = [self.face[d] if d in on else self.cent[d] for d in range(3)]
        z, y, x = torch.meshgrid(c[2], c[1], c[0], indexing="ij")
        return x, y, z


def _modes(gen, base, amp, x, y, z, k=1.0, z_on=False):
    """A constant plus three seeded Fourier modes of amplitude about `amp`."""
    out = torch.full_like(x, base)
    for _ in range(3):
        m = torch.randint(1, 3, (3,), generator=gen).tolist()
        ph = 2 * math.pi * torch.rand(1, generator=gen).item()
        a = amp * (0.5 + torch.rand(1, generator=gen).item())
        out = out + a * torch.sin(k * (m[0] * x + m[1] * y + (m[2] * z if z_on else 0.0)) + ph)
    return out


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _uniform(gen, lo, hi):
    return lo + (hi - lo) * torch.rand(1, generator=gen).item()


def _tube(n, gen):
    """The paper's resistive shock tube (B^x = 1/2, B^y = +-1, rho and p jumping at x = 0,
    Gamma = 2) with seeded resistivity and transverse velocity and field."""
    p = _Problem()
    p.axes(1, n, -0.5, 0.5, "outflow", 2.0)
    x, _, _ = p.mesh()
    left = x < 0.0
    vals = [[_uniform(gen, -0.2, 0.2) for _ in range(4)] for _ in range(2)]
    pick = lambda a, b: torch.where(left, torch.full_like(x, a), torch.full_like(x, b))  # noqa: E731
    v = [pick(vals[0][i], vals[1][i]) for i in range(3)]
    B = [torch.full_like(x, 0.5), pick(1.0, -1.0), pick(vals[0][3], vals[1][3])]
    W = 1.0 / torch.sqrt(1.0 - (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]))
    E = [-e for e in _cross(v, B)]
    p.prim = [pick(1.0, 0.125)] + [W * a for a in v] + [pick(1.0, 0.1)] + E
    p.bface = B
    p.eta_u = 10.0 ** _uniform(gen, -4.0, -2.0)
    return p


def _vortex(n, divb, gen, eta_range=(-5.0, -2.0)):
    """The resistive relativistic Orszag-Tang vortex on periodic [0, 2 pi]^2 with seeded
    phases and resistivity, a guide field and small seeded modes in every field."""
    p = _Problem()
    p.divb = divb
    p.axes(2, n, 0.0, 2 * math.pi, "periodic", 4.0 / 3.0)
    px, py = (2 * math.pi * torch.rand(1, generator=gen).item() for _ in range(2))
    x, y, z = p.mesh()
    state = gen.get_state()
    v = [-0.5 * torch.sin(y + py), 0.5 * torch.sin(x + px), torch.zeros_like(x)]
    v = [a + _modes(gen, 0.0, 0.03, x, y, z) for a in v]
    rho = _modes(gen, 1.0, 0.05, x, y, z)
    pres = _modes(gen, 1.0, 0.05, x, y, z)
    pot = torch.randint(0, 1 << 30, (1,), generator=gen).item()

    def potential(c, on):
        xx, yy, zz = p.mesh(on)
        g = torch.Generator().manual_seed(pot + c)
        a = _modes(g, 0.0, 0.03, xx, yy, zz)
        return a + (torch.cos(yy + py) + 0.5 * torch.cos(2 * (xx + px)) if c == 2 else 0.0)

    # faces (CT) or cells (GLM) of q_B from the potential, and a uniform guide field
    B = [-torch.sin(y + py), torch.sin(2 * (x + px)), torch.full_like(x, 0.2)]
    if divb == "glm":
        g = torch.Generator().manual_seed(pot)
        p.bface = [b + _modes(g, 0.0, 0.05, x, y, z) for b in B]
        p.phi = _modes(g, 0.0, 0.05, x, y, z)
        p.kappa = 1.0
        B = p.bface
    else:
        A = [potential(c, [d for d in range(2) if d != c]) for c in range(3)]
        p.bface = [torch.zeros_like(x) for _ in range(3)]
        up = lambda a, d: torch.roll(a, -1, 2 - d)  # noqa: E731  (the last padded layer is replaced below)
        cb = [(up(A[2], 1) - A[2]) / p.dx[1], -(up(A[2], 0) - A[2]) / p.dx[0],
              (up(A[1], 0) - A[1]) / p.dx[0] - (up(A[0], 1) - A[0]) / p.dx[1]]
        i = [(torch.arange(p.n[d] + 4, device=DEVICE) - 2) % p.n[d] + 2 for d in range(2)]
        p.bface = [b[:, i[1]][:, :, i[0]].contiguous() for b in cb]
        p.bface[2] += 0.2
    W = 1.0 / torch.sqrt(1.0 - (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]))
    p.prim = [rho] + [W * a for a in v] + [pres] + [-e for e in _cross(v, B)]
    gen.set_state(state)
    p.eta_u = 10.0 ** _uniform(gen, *eta_range)
    return p


def _star(n, gen):
    """The magnetised n = 1 polytrope on a fixed conformally flat metric, [-20, 20]^3, with
    an atmosphere, a seeded field strength, resistivity and velocity perturbation."""
    p = _Problem()
    L, K, gamma, rho_c, M = 20.0, 100.0, 2.0, 1.28e-3, 1.4
    p.axes(3, n, -L, L, "outflow", gamma)
    R = math.pi * math.sqrt(K / (2 * math.pi))
    p.rho_atm = rho_c * 1e-10
    p.p_atm = K * p.rho_atm ** gamma
    p_c = K * rho_c ** gamma

    def rho_of(r):
        xi = (math.pi / R) * r
        return torch.where(r < R, torch.clamp(rho_c * torch.sinc(xi / math.pi), min=p.rho_atm),
                           torch.full_like(r, p.rho_atm))

    x, y, z = p.mesh()
    r = torch.sqrt(x * x + y * y + z * z)
    rbar = torch.sqrt(r * r + 4 * M * M)
    p.alpha = 1.0 - 2.0 * M / (rbar + M)
    p.psi = 1.0 + M / (2.0 * rbar)
    rho = rho_of(r)
    u = [(rho / rho_c) * _modes(gen, 0.0, 0.01, x, y, z, k=2 * math.pi / L, z_on=True) for _ in range(3)]
    zero = torch.zeros_like(x)
    p.prim = [rho] + u + [K * rho ** gamma, zero, zero.clone(), zero.clone()]
    A_b = math.sqrt(2.0 * 10.0 ** _uniform(gen, -3.5, -2.5) * p_c) / (2.0 * 0.96 * p_c)

    def fpot(xx, yy, zz):
        return A_b * torch.clamp(K * rho_of(torch.sqrt(xx * xx + yy * yy + zz * zz)) ** gamma - 0.04 * p_c, min=0.0)

    xa, ya, za = p.mesh([1, 2])
    xb, yb, zb = p.mesh([0, 2])
    p.A = [-ya * fpot(xa, ya, za), xb * fpot(xb, yb, zb), torch.zeros_like(x)]
    p.eta_u = 10.0 ** _uniform(gen, -6.0, -5.0)
    p.eta = torch.where(r < R, torch.full_like(r, p.eta_u), torch.ones_like(r))
    return p


def _problems(case, seed):
    gen = torch.Generator().manual_seed(int(seed))
    kind = case["kind"]
    if kind == "tube":
        return [_tube(case["n"], gen)]
    if kind == "vortex":
        return [_vortex(case["n"], case["divb"], gen)]
    if kind == "star":
        return [_star(case["n"], gen)]
    if kind == "batch":
        return [_vortex(n, "ct", gen, (-6.0, 0.0)) for n in _sides(case)]
    p = _vortex(case["n"], "ct", gen)
    noise = torch.Generator(device=DEVICE).manual_seed(int(seed) + 1)
    p.bface = [b + 0.05 * torch.randn(b.shape, dtype=b.dtype, device=DEVICE, generator=noise) for b in p.bface]
    return [p]


def _sides(case):
    """The sides of a batch's boxes: spread evenly over [lo, hi], in a mixed order."""
    k, lo, hi = case["boxes"], case["lo"], case["hi"]
    return [lo + round((hi - lo) * ((7 * i + case["mix"]) % k) / max(k - 1, 1)) for i in range(k)]


_RUN_STEPS = {"tube": 400, "vortex": 1000, "batch": 1000, "star": 100, "clean": 1000}


class _State:
    pass


def _start(s):
    for sol, p in zip(s.solvers, s.problems):
        sol.init_from_prims(p.prim, A_edge=p.A, bface=p.bface, phi=p.phi)
    s.left = s.steps


def prepare(case, seed):
    from paper_2110_03732_gb300 import grmhd

    s = _State()
    s.problems = _problems(case, seed)
    s.solvers = []
    for p in s.problems:
        sol = grmhd.Solver(p.ndim, p.n, p.lo, p.hi, [p.bc] * 3, p.gamma, p.cfl, device=DEVICE, rho_atm=p.rho_atm,
                           p_atm=p.p_atm, precision=case["precision"], rec=case["rec"], divb=p.divb, kappa=p.kappa)
        sol.set_metric(p.alpha, p.psi)
        sol.set_eta(p.eta, p.eta_u)
        s.solvers.append(sol)
    s.steps = _RUN_STEPS[case["kind"]]
    _start(s)
    s.batch = s.cycles = None
    s.dt = [sol.compute_dt() for sol in s.solvers]
    if case["kind"] == "batch":
        s.batch = grmhd.Batch(s.solvers)
        s.batch.set_dt(s.dt)
    if case["kind"] == "clean":
        s.cycles = case["cycles"]
    return s


def _interior(sol):
    return tuple(slice(sol.ng[d], sol.ng[d] + sol.grid.n[d]) for d in (2, 1, 0))


def run(s):
    if s.left == 0:   # the run is over: the next one begins from the initial data
        _start(s)
    s.left -= 1
    if s.batch is not None:
        s.batch.step()
        return [sol.state[(slice(None),) + _interior(sol)] for sol in s.solvers]
    sol = s.solvers[0]
    if s.cycles is not None:
        sol.clean_divb(s.cycles)
        return [b[_interior(sol)] for b in sol.bf]
    sol.step(s.dt[0])
    return [t[_interior(sol)] for t in sol.state]


def work(case):
    """Bytes: the state read and written once, the metric and resistivity read.  Flops:
    those of the method per cell and stage (residual of the implicit solve, flux and
    reconstruction per face, EMF per edge, sources and update)."""
    kind = case["kind"]
    if kind == "clean":
        cells = case["n"] ** 2
        # a V(2,2) cycle: four sweeps, residual, interpolation; 4/3 for the levels
        return {"bytes": 8 * 4 * cells, "flops": case["cycles"] * cells * 4 / 3 * (4 * 6 + 8 + 10)}
    if kind == "tube":
        ndim, cells = 1, case["n"]
    elif kind == "star":
        ndim, cells = 3, case["n"] ** 3
    else:
        ndim, cells = 2, case["n"] ** 2 if kind == "vortex" else sum(n * n for n in _sides(case))
    edges = {1: 0, 2: 1, 3: 3}[ndim]
    arrays = 22 + (2 if case.get("divb") == "glm" else 0) + (3 if kind == "star" else 0)
    return {"bytes": 8 * arrays * cells, "flops": 2 * cells * (130 + 230 * ndim + 60 * edges + 60 + 35 * ndim)}


# --------------------------------------------------------------------------
# one IMEX-SSP2 step in plain torch (arXiv 2110.03732), 64 bits
# --------------------------------------------------------------------------

def _ext(p, a, face=None):
    """Interior and three mapped ghost layers per active direction; `face`: the direction
    whose lower faces `a` lives on (one more layer there)."""
    for d in range(p.ndim):
        n = p.n[d]
        m = torch.arange(-3, n + 3 + (d == face), device=a.device)
        m = m % n if p.bc == "periodic" else m.clamp(0, n if d == face else n - 1)
        a = a.index_select(2 - d, m + 2)
    return a


def _metric_ext(p, a):
    """A metric array with its stored ghosts, three layers deep."""
    if a is None:
        return torch.ones((), dtype=torch.float64, device=DEVICE).expand([1 if d >= p.ndim else p.n[d] + 6 for d in (2, 1, 0)])
    for d in range(p.ndim):
        a = a.index_select(2 - d, torch.arange(-1, p.n[d] + 5, device=a.device).clamp(0, p.n[d] + 3))
    return a


def _in(p, a, keep=(), upper=()):
    """The interior of an extended array, all layers of the directions in `keep` and one
    more in `upper`."""
    for d in range(p.ndim):
        if d not in keep:
            a = a.narrow(2 - d, 3, p.n[d] + (d in upper))
    return a


def _recon(x, axis, ppm):
    """Left and right states at the n + 1 faces from n + 6 cells along `axis`."""
    n = x.shape[axis] - 6
    s = lambda a, i, k: a.narrow(axis, i, k)  # noqa: E731
    d = s(x, 1, n + 5) - s(x, 0, n + 5)
    dm, dp = s(d, 0, n + 4), s(d, 1, n + 4)
    zero = torch.zeros((), dtype=x.dtype, device=x.device)
    top, bot = torch.maximum(torch.minimum(dm, dp), zero), torch.minimum(torch.maximum(dm, dp), zero)
    hs = torch.minimum(torch.maximum(0.25 * (s(x, 2, n + 4) - s(x, 0, n + 4)), bot), top)   # cells 1..n+4
    c = s(x, 1, n + 4)
    if not ppm:
        return s(c + hs, 1, n + 1), s(c - hs, 2, n + 1)
    face = s(c, 0, n + 3) + 0.5 * (s(c, 1, n + 3) - s(c, 0, n + 3)) - (2 * s(hs, 1, n + 3) - 2 * s(hs, 0, n + 3)) / 6
    a0, aL, aR = s(c, 1, n + 2), s(face, 0, n + 2), s(face, 1, n + 2)
    flat = (aR - a0) * (a0 - aL) <= 0
    dd, m6 = aR - aL, 6 * (a0 - 0.5 * (aL + aR))
    nL = torch.where(flat, a0, torch.where(dd * m6 > dd * dd, 3 * a0 - 2 * aR, aL))
    nR = torch.where(flat, a0, torch.where(-dd * dd > dd * m6, 3 * a0 - 2 * aL, aR))
    return s(nR, 0, n + 1), s(nL, 1, n + 1)


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _conserved(p, rho, u, pr, E, B):
    """D, S, tau and W, U, rho h of orthonormal-frame primitives."""
    W = torch.sqrt(1.0 + _dot(u, u))
    h = rho + p.gamma / (p.gamma - 1.0) * pr
    U = 0.5 * (_dot(E, E) + _dot(B, B))
    x = _cross(E, B)
    return rho * W, [h * W * u[i] + x[i] for i in range(3)], h * W * W - pr + U - rho * W, W, U, h


def _fluxes(p, prim, Bcell, Bnorm, psi, alp, d, ppm, phi=None):
    """Twice the HLL flux at the d-faces (speeds alpha / psi^2), 8 variables, or 12 (GLM)."""
    ax = 2 - d
    f0 = 3
    mean = lambda a: 0.5 * (a.narrow(ax, f0 - 1, p.n[d] + 1) + a.narrow(ax, f0, p.n[d] + 1))  # noqa: E731
    ps, al = mean(_in(p, psi, [d])), mean(_in(p, alp, [d]))
    p2 = ps * ps
    rec = [_recon(_in(p, v, [d]), ax, ppm) for v in prim]
    rB = [_recon(_in(p, b, [d]), ax, ppm) if (phi is not None or e != d) else None for e, b in enumerate(Bcell)]
    rphi = _recon(_in(p, phi, [d]), ax, ppm) if phi is not None else None
    sides = []
    for k in range(2):
        rho, pr = rec[0][k], rec[4][k]
        u, E = [p2 * rec[1 + i][k] for i in range(3)], [p2 * rec[5 + i][k] for i in range(3)]
        B = [p2 * rB[e][k] if rB[e] is not None else Bnorm / (p2 * p2) for e in range(3)]
        D, S, tau, W, U, h = _conserved(p, rho, u, pr, E, B)
        q = [p2 ** 3 * D] + [p2 ** 4 * s for s in S] + [p2 ** 3 * tau] + [p2 ** 2 * e for e in E]
        f = [p2 ** 2 * al * rho * u[d]]
        for j in range(3):
            f.append(p2 ** 3 * al * (h * u[d] * u[j] - E[d] * E[j] - B[d] * B[j] + (pr + U if j == d else 0.0)))
        f.append(p2 ** 2 * al * (S[d] - rho * u[d]))
        fE = [None] * 3
        fE[d] = torch.zeros_like(rho)
        fE[(d + 1) % 3], fE[(d + 2) % 3] = al * p2 * B[(d + 2) % 3], -al * p2 * B[(d + 1) % 3]
        f += fE
        if phi is not None:
            Ec = [rec[5 + i][k] for i in range(3)]
            qB = [p2 ** 3 * rB[e][k] for e in range(3)]
            fB = [None] * 3
            fB[d] = torch.zeros_like(rho)
            fB[(d + 1) % 3], fB[(d + 2) % 3] = -al * p2 ** 2 * Ec[(d + 2) % 3], al * p2 ** 2 * Ec[(d + 1) % 3]
            q += qB + [p2 ** 3 * rphi[k]]
            f += fB + [al * qB[d]]
        sides.append((q, f))
    (qL, fL), (qR, fR) = sides
    c = al / p2
    return [a + b - c * (y - x) for a, b, x, y in zip(fL, fR, qL, qR)]


def _emf(p, prim, bf, psi, alp, c, ppm):
    """Upwind edge EMF along c, on the lower edges and one more in the transverse directions."""
    a, b = (c + 1) % 3, (c + 2) % 3
    aa, ba = a < p.ndim, b < p.ndim
    trans = [d for d in (a, b) if d < p.ndim]
    n = p.n
    e = _in(p, psi ** 4 * prim[5 + c], trans)
    EA = _recon(e, 2 - a, ppm) if aa else (e, e)
    EXY = [_recon(x, 2 - b, ppm) if ba else (x, x) for x in EA]
    lo = lambda x, d, off: x.narrow(2 - d, 3 + off, n[d] + 1) if d < p.ndim else x  # noqa: E731
    qb = lo(_in(p, bf[b], trans), b, 0)
    qa = lo(_in(p, bf[a], trans), a, 0)
    zero = torch.zeros((), dtype=torch.float64, device=DEVICE)
    jb = (lambda r: r[1] - r[0])(_recon(qb.narrow(2 - a, 0, n[a] + 6), 2 - a, ppm)) if aa else zero
    ja = (lambda r: r[1] - r[0])(_recon(qa.narrow(2 - b, 0, n[b] + 6), 2 - b, ppm)) if ba else zero
    ps, al = _in(p, psi, trans), _in(p, alp, trans)
    at = lambda x, oa, ob: lo(lo(x, a, oa), b, ob)  # noqa: E731
    offs = [(i, j) for i in ((0, -1) if aa else (0,)) for j in ((0, -1) if ba else (0,))]
    ale = sum(at(al, i, j) for i, j in offs) / len(offs)

    def speed(d, other):
        if d >= p.ndim:
            return zero + 1.0
        best = None
        for o in (0, -1) if other < p.ndim else (0,):
            pick = (lambda x, k: at(x, k, o)) if d == a else (lambda x, k: at(x, o, k))
            s = 0.5 * (pick(al, 0) + pick(al, -1)) / (0.5 * (pick(ps, 0) + pick(ps, -1))) ** 2
            best = s if best is None else torch.maximum(best, s)
        return best

    mean = 0.25 * (EXY[0][0] + EXY[0][1] + EXY[1][0] + EXY[1][1])
    return ale * mean + 0.5 * speed(a, b) * jb - 0.5 * speed(b, a) * ja


def _explicit(p, prim, bf, phi, ppm):
    """The explicit operator L of the cell variables (8, or 12 for GLM) and of the faces."""
    glm = p.divb == "glm"
    psi, alp = _metric_ext(p, p.psi), _metric_ext(p, p.alpha)
    P = [_ext(p, v) for v in prim]
    bx = [_ext(p, b, None if glm else d) for d, b in enumerate(bf)]
    mid = lambda b, d: 0.5 * (b.narrow(2 - d, 0, p.n[d] + 6) + b.narrow(2 - d, 1, p.n[d] + 6))  # noqa: E731
    qc = [b if glm or d >= p.ndim else mid(b, d) for d, b in enumerate(bx)]
    if not glm and p.bc == "outflow":
        qc = [_ext(p, _pad_mid(p, b, d)) for d, b in enumerate(bf)]
    Bc = [q / psi ** 6 for q in qc]
    qphi = _ext(p, phi) if glm else None
    L = [0.0] * (12 if glm else 8)
    for d in range(p.ndim):
        bn = None if glm else _in(p, bx[d], [d]).narrow(2 - d, 3, p.n[d] + 1)
        F = _fluxes(p, P, Bc, bn, psi, alp, d, ppm, qphi / psi ** 6 if glm else None)
        for v, f in enumerate(F):
            L[v] = L[v] - (f.narrow(2 - d, 1, p.n[d]) - f.narrow(2 - d, 0, p.n[d])) * (0.5 / p.dx[d])
    # non-stiff sources
    ps, al = _in(p, psi), _in(p, alp)
    p2 = ps * ps
    diff = lambda x, d: (_in(p, x, [d]).narrow(2 - d, 4, p.n[d]) - _in(p, x, [d]).narrow(2 - d, 2, p.n[d])) * (0.5 / p.dx[d])  # noqa: E731
    I = [_in(p, v) for v in P]
    u, E = [p2 * I[1 + i] for i in range(3)], [p2 * I[5 + i] for i in range(3)]
    B = [p2 * _in(p, b) for b in Bc]
    D, S, tau, W, U, h = _conserved(p, I[0], u, I[4], E, B)
    div = sum(diff(psi ** 6 * P[5 + d], d) for d in range(p.ndim))
    for i in range(3):
        L[5 + i] = L[5 + i] - al * div * I[1 + i] / W
    if p.alpha is not None:
        tr = h * _dot(u, u) + 3 * I[4] + U
        for i in range(p.ndim):
            da, dp = diff(alp, i), diff(psi, i)
            L[1 + i] = L[1 + i] + p2 ** 3 * (-(tau + D) * da + 2 * al * (dp / ps) * tr)
            L[4] = L[4] - p2 ** 2 * S[i] * da
    if glm:
        L[11] = L[11] - al * p.kappa * _in(p, qphi)
        for d in range(p.ndim):
            L[8 + d] = L[8 + d] - al * p2 * diff(qphi / psi ** 6, d)
            if p.alpha is not None:
                L[11] = L[11] + _in(p, bx[d]) * diff(alp, d)
        return L
    emf = [_emf(p, P, bx, psi, alp, c, ppm) if any(d != c for d in range(p.ndim)) else None for c in range(3)]
    step = lambda e, d: (e.narrow(2 - d, 1, p.n[d]) - e.narrow(2 - d, 0, p.n[d])) / p.dx[d]  # noqa: E731
    for fa in range(3):
        fb, fc = (fa + 1) % 3, (fa + 2) % 3
        r = 0.0
        if fb < p.ndim:
            r = r - step(emf[fc], fb)
        if fc < p.ndim:
            r = r + step(emf[fb], fc)
        L.append(r)
    return L


def _pad_mid(p, b, d):
    """Cell means of a padded face array (outflow grids), on the padded cells."""
    if d >= p.ndim:
        return b
    return torch.cat([0.5 * (b.narrow(2 - d, 0, b.shape[2 - d] - 1) + b.narrow(2 - d, 1, b.shape[2 - d] - 1)),
                      b.narrow(2 - d, b.shape[2 - d] - 1, 1)], 2 - d)


def _solve(p, q, qb, u0, a_dt):
    """Implicit E and velocity (Newton in the orthonormal frame): primitives and the rate R."""
    pad = tuple(slice(2 if d < p.ndim else 0, (2 if d < p.ndim else 0) + p.n[d]) for d in (2, 1, 0))
    one = torch.ones_like(q[0])
    ps = p.psi[pad] if p.psi is not None else one
    al = p.alpha[pad] if p.alpha is not None else one
    eta = p.eta[pad] if p.eta is not None else p.eta_u * one
    p2 = ps * ps
    D, S, tau = q[0] / p2 ** 3, [q[1 + i] / p2 ** 4 for i in range(3)], q[4] / p2 ** 3
    Es, B = [q[5 + i] / p2 ** 2 for i in range(3)], [b / p2 ** 2 for b in qb]
    et = eta / (al * a_dt)
    ig = (p.gamma - 1.0) / p.gamma
    shape = D.shape
    atm = D < 10.0 * p.rho_atm if p.rho_atm > 0 else torch.zeros(shape, dtype=torch.bool, device=D.device)
    sel = ~atm
    D_, tau_, et_ = D[sel], tau[sel], et[sel]
    S_, Es_, B_ = [s[sel] for s in S], [e[sel] for e in Es], [b[sel] for b in B]
    u = [x[sel] for x in u0]

    def residual(u):
        W = torch.sqrt(1.0 + _dot(u, u))
        A1, A0, Eu, uB = et_ / (1.0 + et_ * W), W + et_, _dot(Es_, u), _cross(u, B_)
        E = [(et_ * Es_[i] + A1 * Eu * u[i] - uB[i]) / A0 for i in range(3)]
        U = 0.5 * (_dot(E, E) + _dot(B_, B_))
        base = tau_ + D_ - U
        den = W * W - ig
        wt = (W * base - D_ * ig) / den
        x = _cross(E, B_)
        f = [wt * u[i] - S_[i] + x[i] for i in range(3)]
        return f, (W, A1, A0, Eu, E, base, den, wt)

    f, aux = residual(u)
    for _ in range(40):
        W, A1, A0, Eu, E, base, den, wt = aux
        J = [[None] * 3 for _ in range(3)]
        for j in range(3):
            dE = [-E[i] * u[j] / W - A1 * A1 * u[j] / W * Eu * u[i] + A1 * Es_[j] * u[i] + (A1 * Eu if i == j else 0.0)
                  for i in range(3)]
            j1, j2 = (j + 1) % 3, (j + 2) % 3
            dE[j1] = dE[j1] + B_[j2]   # -(e_j x B)
            dE[j2] = dE[j2] - B_[j1]
            dE = [x / A0 for x in dE]
            dw = (u[j] / W * base - W * _dot(E, dE) - 2 * wt * u[j]) / den
            x = _cross(dE, B_)
            for i in range(3):
                J[i][j] = u[i] * dw + x[i] + (wt if i == j else 0.0)
        cof = [_cross(J[1], J[2]), _cross(J[2], J[0]), _cross(J[0], J[1])]   # rows: cofactors of row i
        det = _dot(J[0], cof[0])
        dx = [-(cof[0][j] * f[0] + cof[1][j] * f[1] + cof[2][j] * f[2]) / det for j in range(3)]
        g0 = _dot(f, f)
        lam = torch.ones_like(g0)
        for _ in range(8):
            un = [u[i] + lam * dx[i] for i in range(3)]
            fn, an = residual(un)
            bad = ~(_dot(fn, fn) <= torch.clamp(g0, min=1e-60)) & (g0 > 1e-28 * _dot(S_, S_))
            if not bool(bad.any()):
                break
            lam = torch.where(bad, 0.5 * lam, lam)
        moved = max((float((lam * x).abs().max()) for x in dx if x.numel()), default=0.0)
        u, f, aux = un, fn, an
        if moved < 1e-16:
            break
    W, wt, E = aux[0], aux[7], aux[4]

    def full(fill, vals):
        out = fill.clone() if torch.is_tensor(fill) else torch.full(shape, fill, dtype=torch.float64, device=D.device)
        out[sel] = vals
        return out

    rho = full(p.rho_atm, D_ / W)
    pr = full(p.p_atm, (wt / W - D_ / W) * ig)
    uu = [full(0.0, x) for x in u]
    EE = [full(Es[i], E[i]) for i in range(3)]
    R = [(p2 ** 2 * EE[i] - q[5 + i]) / a_dt for i in range(3)]
    return [rho] + [x / p2 for x in uu] + [pr] + [e / p2 for e in EE], R


def _exact_step(p, ppm, dt):
    """The state after one IMEX-SSP2 step: 8 conserved variables, 3 fields, (q_Phi)."""
    glm = p.divb == "glm"
    pad = tuple(slice(2 if d < p.ndim else 0, (2 if d < p.ndim else 0) + p.n[d]) for d in (2, 1, 0))
    bf = p.bface
    if p.A is not None:
        bf = []
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            r = torch.zeros_like(p.A[0])
            if b < p.ndim:
                r = r + (torch.roll(p.A[c], -1, 2 - b) - p.A[c]) / p.dx[b]
            if c < p.ndim:
                r = r - (torch.roll(p.A[b], -1, 2 - c) - p.A[b]) / p.dx[c]
            bf.append(r)
    bf = [b.clone() for b in bf]
    one = torch.ones_like(p.prim[0])[pad]
    ps = p.psi[pad] if p.psi is not None else one
    p2 = ps * ps

    def cells(b):
        if glm:
            return [x[pad] for x in b]
        out = []
        for d in range(3):
            if d >= p.ndim:
                out.append(b[d][pad])
                continue
            e = _in(p, _ext(p, b[d], d), [d])
            out.append(0.5 * (e.narrow(2 - d, 3, p.n[d]) + e.narrow(2 - d, 4, p.n[d])))
        return out

    pr = [v[pad] for v in p.prim]
    B = [x / p2 ** 2 for x in cells(bf)]
    D, S, tau, _, _, _ = _conserved(p, pr[0], [p2 * x for x in pr[1:4]], pr[4], [p2 * x for x in pr[5:8]], B)
    q = [p2 ** 3 * D] + [p2 ** 4 * s for s in S] + [p2 ** 3 * tau] + [p2 ** 3 * x for x in pr[5:8]]
    qphi = None
    if glm:
        full = p.psi if p.psi is not None else torch.ones_like(p.phi)
        qphi = full ** 6 * p.phi
    g = 1.0 - 1.0 / math.sqrt(2.0)
    u = [p2 * x for x in pr[1:4]]
    qs, bs, phs = q, bf, qphi
    Ls, Rs = [], []
    for stage in range(2):
        prim, R = _solve(p, qs, cells(bs), u, g * dt)
        u = [p2 * x for x in prim[1:4]]
        padded = []
        for v, x in zip(p.prim, prim):
            y = v.clone()
            y[pad] = x
            padded.append(y)
        L = _explicit(p, padded, bs, phs, ppm)
        Ls.append(L)
        Rs.append(R)
        if stage == 0:
            qs = [q[v] + dt * (L[v] + ((1 - 2 * g) * R[v - 5] if v >= 5 else 0.0)) for v in range(8)]
            bs = [b.clone() for b in bf]
            for d in range(3):
                if glm:
                    bs[d][pad] += dt * L[8 + d]
                elif torch.is_tensor(L[8 + d]):
                    _faces(p, bs[d], d).add_(dt * _faces_of(p, L[8 + d], d))
            if glm:
                phs = qphi.clone()
                phs[pad] += dt * L[11]
    out = [q[v] + 0.5 * dt * (Ls[0][v] + Ls[1][v] + (Rs[0][v - 5] + Rs[1][v - 5] if v >= 5 else 0.0)) for v in range(8)]
    for d in range(3):
        b = bf[d].clone()
        if glm:
            b[pad] += 0.5 * dt * (Ls[0][8 + d] + Ls[1][8 + d])
        elif torch.is_tensor(Ls[0][8 + d]):
            _faces(p, b, d).add_(0.5 * dt * _faces_of(p, Ls[0][8 + d] + Ls[1][8 + d], d))
        out.append(b[pad])
    if glm:
        out.append(qphi[pad] + 0.5 * dt * (Ls[0][11] + Ls[1][11]))
    return out


def _faces(p, b, fd):
    """The faces of a padded array that a step updates (the upper boundary face too where
    the direction is not periodic)."""
    for d in range(p.ndim):
        b = b.narrow(2 - d, 2, p.n[d] + (1 if d == fd and p.bc != "periodic" else 0))
    return b


def _faces_of(p, r, fd):
    return r.narrow(2 - fd, 0, p.n[fd]) if fd < p.ndim and p.bc == "periodic" else r


def _time_step(p):
    if p.alpha is None:
        return p.cfl / sum(1.0 / p.dx[d] for d in range(p.ndim))
    pad = tuple(slice(2, 2 + p.n[d]) for d in (2, 1, 0))
    return p.cfl / float((p.alpha[pad] / p.psi[pad] ** 2).max() * sum(1.0 / p.dx[d] for d in range(p.ndim)))


def exact(case, seed):
    out = []
    for p in _problems(case, seed):
        if case["kind"] == "clean":
            return _exact_clean(p)
        out.append(_exact_step(p, case["rec"] == "ppm", _time_step(p)))
    return [torch.stack(s) for s in out] if case["kind"] == "batch" else out[0]


def _exact_clean(p):
    """The staggered field less the gradient of the exact solution of the compact Poisson
    problem (periodic, by Fourier transform)."""
    b = [x[:, 2:-2, 2:-2] for x in p.bface]
    div = (torch.roll(b[0], -1, 2) - b[0]) / p.dx[0] + (torch.roll(b[1], -1, 1) - b[1]) / p.dx[1]
    k = [2.0 - 2.0 * torch.cos(2 * math.pi * torch.arange(p.n[d], dtype=torch.float64, device=DEVICE) / p.n[d])
         for d in range(2)]
    lam = -(k[1][:, None] / p.dx[1] ** 2 + k[0][None, :] / p.dx[0] ** 2)
    lam[0, 0] = 1.0
    f = torch.fft.fft2(div[0]) / lam
    f[0, 0] = 0.0
    phi = torch.fft.ifft2(f).real[None]
    return [b[0] - (phi - torch.roll(phi, 1, 2)) / p.dx[0], b[1] - (phi - torch.roll(phi, 1, 1)) / p.dx[1], b[2]]
