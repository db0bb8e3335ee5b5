"""One and two V(2,2) cycles of the multigrid cleaning (csrc/elliptic.cu), field by field
against the same cycle in plain NumPy: red-black Gauss-Seidel (two sweeps down from zero, two
up), the mean of the children's residuals, linear interpolation (3/4, 1/4 per direction), and the
coarsest level solved exactly.  A leg that smooths, restricts or interpolates otherwise differs
at once, though it would converge to the same field.

Tolerance 1e-11 of the field's scale: the coarsest solve stops at 1e-15 of its right-hand
side, which its smallest eigenvalue (a thousandth of the largest at 35^2) magnifies to 1e-12.
(Long thin grids between closed ends are left to the test of the converged field: on a
coarsest level of 2 x 512 cells that ratio is 2e5, and conjugate gradients end at 1e-8.)"""
import numpy as np
import pytest

from paper_2110_03732_gb300 import problems as P
from parity_tools import check

torch = pytest.importorskip("torch")
sp = pytest.importorskip("scipy.sparse")
spla = pytest.importorskip("scipy.sparse.linalg")
pytestmark = pytest.mark.gpu

CASES = [
    ([72, 40], "outflow"),       # tiles of 16, 8 left over each way
    ([72, 40], "periodic"),
    ([1024, 4], "periodic"),     # a wrapped extent shorter than a tile's halo
    ([40, 72], "outflow"),
    ([656, 240], "outflow"),
    ([1040, 528], "outflow"),    # tiles of 32 (549120 cells), half a tile left over
    ([1040, 528], "periodic"),
    ([70, 70], "periodic"),      # a coarsest level of 35^2, in global memory
    ([560, 560], "outflow"),
    ([96, 64], "periodic"),      # a coarsest level of 3 x 2 for one warp
    ([200, 200], "outflow"),     # 25^2
    ([112, 112], "outflow"),     # 7^2: lanes of the warp with one and two cells
]


def shift(a, ax, s, bc):
    """The neighbour's value along an axis (0 past a boundary) and whether there is one."""
    r, there = np.roll(a, -s, ax), np.ones(a.shape, bool)
    if bc != "periodic":
        sl = [slice(None)] * 2
        sl[ax] = -1 if s > 0 else 0
        r = r.copy()
        r[tuple(sl)] = 0.0
        there[tuple(sl)] = False
    return r, there


def stencil(phi, ih2, bc):
    nb, diag = np.zeros_like(phi), np.zeros_like(phi)
    for ax in (0, 1):
        for s in (-1, 1):
            v, there = shift(phi, ax, s, bc)
            nb += v * ih2[ax]
            diag += there * ih2[ax]
    return nb, diag


def smooth(phi, rhs, ih2, bc):
    color = np.add.outer(np.arange(phi.shape[0]), np.arange(phi.shape[1])) & 1
    for s in (0, 1, 0, 1):
        nb, diag = stencil(phi, ih2, bc)
        phi = np.where(color == s, (nb - rhs) / diag, phi)
    return phi


def interpolate(c, bc):
    for ax in (0, 1):
        wide = np.take(c, np.clip(np.arange(-1, c.shape[ax] + 1), 0, c.shape[ax] - 1), ax)
        if bc == "periodic":
            wide = np.take(c, np.arange(-1, c.shape[ax] + 1) % c.shape[ax], ax)
        n = c.shape[ax]
        lo, mid, hi = (np.take(wide, np.arange(k, k + n), ax) for k in range(3))
        c = np.stack([0.75 * mid + 0.25 * lo, 0.75 * mid + 0.25 * hi], ax + 1)
        shape = [mid.shape[0], mid.shape[1]]
        shape[ax] *= 2
        c = c.reshape(shape)
    return c


def coarsest(rhs, ih2, bc):
    n = rhs.size
    idx = np.arange(n).reshape(rhs.shape)
    A = sp.lil_matrix((n, n))
    for ax in (0, 1):
        for s in (-1, 1):
            j, there = shift(idx, ax, s, bc)
            for a, b in zip(idx[there], j[there]):
                A[a, b] += ih2[ax]
                A[a, a] -= ih2[ax]
    b = (rhs - rhs.mean()).ravel()
    A[0, :] = 0.0   # (the constant is free: pin one cell, then take the mean out)
    A[0, 0] = 1.0
    b[0] = 0.0
    x = spla.spsolve(A.tocsc(), b).reshape(rhs.shape)
    return x - x.mean()


def cycle(phi, rhs, ih2, bc):
    if any(k % 2 or k < 4 for k in rhs.shape):
        return coarsest(rhs, ih2, bc)
    phi = smooth(phi, rhs, ih2, bc)
    nb, diag = stencil(phi, ih2, bc)
    res = rhs - (nb - diag * phi)
    ny, nx = rhs.shape
    res = res.reshape(ny // 2, 2, nx // 2, 2).mean(axis=(1, 3))
    c = cycle(np.zeros_like(res), res, [h / 4 for h in ih2], bc)
    return smooth(phi + interpolate(c, bc), rhs, ih2, bc)


@pytest.mark.parametrize("n,bc", CASES)
@pytest.mark.parametrize("cycles", [1, 2])
def test_cycles_match_numpy(n, bc, cycles):
    from paper_2110_03732_gb300 import build, grmhd
    build.build()
    pr = P.random_box(91, 2, n, bc=bc)
    pr.hi = [n[0] / 64.0, n[1] / 48.0, 1.0]
    S = grmhd.Solver.from_problem(pr)
    rng = np.random.default_rng(5)
    q = [rng.normal(size=(n[1] + 4, n[0] + 4)) for _ in range(2)]
    for d in range(2):
        S.bf[d].copy_(torch.as_tensor(q[d][None], device="cuda"))
    S.clean_divb(cycles)
    got = [S.bf[d].cpu().numpy()[0, 2:-2, 2:-2] for d in range(2)]
    idx = [64.0, 48.0]
    face = [q[0][2:-2, 2:-1], q[1][2:-1, 2:-2]]   # lower faces of the cells and the last upper one
    if bc == "periodic":
        face = [np.concatenate([face[0][:, :-1], face[0][:, :1]], 1), np.concatenate([face[1][:-1], face[1][:1]], 0)]
    div = np.diff(face[0], axis=1) * idx[0] + np.diff(face[1], axis=0) * idx[1]
    rhs = div - div.mean()
    ih2 = [idx[1] ** 2, idx[0] ** 2]
    phi = np.zeros_like(rhs)
    for _ in range(cycles):
        phi = cycle(phi, rhs, ih2, bc)
    for d, ax in ((0, 1), (1, 0)):
        low, there = shift(phi, ax, -1, bc)
        want = q[d][2:-2, 2:-2] - np.where(there, (phi - low) * idx[d], 0.0)
        check(got[d], want, (n, bc, d), 1e-11, 1e-11)
