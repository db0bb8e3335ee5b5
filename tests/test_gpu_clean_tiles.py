"""The tiled legs of the 2-D multigrid cleaning (csrc/elliptic.cu) at the sizes where a tile
can go wrong: extents that are not multiples of the tile (16, and 32 on large levels),
periodic extents shorter than a tile's halo, and non-periodic boundaries inside a tile.
The cleaned field is compared with the oracle's exact solve of the same discrete problem,
relative L1 <= 1e-10 per component once the V-cycles have converged, as for the other
levels."""
import numpy as np
import pytest

import oracle
from oracle import elliptic as E
from paper_2110_03732_gb300 import problems as P
from parity_tools import check

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    ([72, 40], "outflow"),      # 8 left over each way, boundaries inside the tiles
    ([72, 40], "periodic"),
    ([1024, 4], "periodic"),    # a wrapped extent shorter than the halo
    ([4, 1024], "outflow"),
    ([656, 240], "outflow"),    # tiles of 32, half a tile left over
    ([656, 240], "periodic"),
]


@pytest.mark.parametrize("n,bc", CASES)
@pytest.mark.parametrize("divb", ["ct", "glm"])
def test_tiled_cleaning_matches_exact_solve(n, bc, divb):
    from paper_2110_03732_gb300 import build, grmhd
    build.build()
    glm = divb == "glm"
    pr = P.random_box(91, 2, n, bc=bc, glm=glm)
    # square cells, whatever the extents
    pr.hi = [n[0] / 64.0, n[1] / 64.0, 1.0]
    S = grmhd.Solver.from_problem(pr, divb=divb)
    g = oracle.Grid(2, pr.n, pr.dx, pr.bc, pr.gamma)
    rng = np.random.default_rng(17)
    fields = [rng.normal(size=g.shape) for _ in range(3)]
    for d in range(3):
        S.bf[d].copy_(torch.as_tensor(fields[d], device="cuda"))
    S.clean_divb(40)
    torch.cuda.synchronize()
    ref, _ = (E.clean_cells if glm else E.clean_faces)(g, fields)
    inside = g.interior()
    for d in range(2):
        check(S.bf[d].cpu().numpy()[inside], ref[d][inside], (n, bc, d))
