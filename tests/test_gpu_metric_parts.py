"""Steps on a metric against the oracle where the FP64 metric code has branches of its own: a lapse
without a conformal factor and the reverse (edge speeds, sources, charge), and a cell whose
implicit solve fails without an atmosphere (its charge comes from the primitives it keeps).
Tolerances as for the other parity tests; in mixed precision 1e-5, as for its other steps."""
import pytest

import oracle
from paper_2110_03732_gb300 import problems as P
from parity_tools import check

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2110_03732_gb300 import build, grmhd
    build.build()
    return grmhd


def compare(S, st, tol, tol_max):
    i = st.grid.interior()
    for v in range(8):
        check(S.q[v].cpu().numpy()[i], st.q[v][i], f"q{v}", tol, tol_max)
    for d in range(3):
        check(S.bf[d].cpu().numpy()[i], st.bf[d][i], f"bf{d}", tol, tol_max)


@pytest.mark.parametrize("part", ["alpha", "psi"])
@pytest.mark.parametrize("ndim,n", [(1, [37]), (2, [27, 22]), (3, [13, 11, 9])])
@pytest.mark.parametrize("rec", ["mc", "ppm"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_lapse_or_conformal_factor_alone(G, part, ndim, n, rec, precision):
    pr = P.random_box(21, ndim, n, bc="outflow", metric=True)
    setattr(pr, "psi" if part == "alpha" else "alpha", None)
    st = oracle.from_problem(pr, rec=rec)
    S = G.Solver.from_problem(pr, rec=rec, precision=precision)
    dt = S.compute_dt()
    for _ in range(2):
        st.step(dt)
        S.step(dt)
    if precision == "fp64":
        compare(S, st, 1e-10, 1e-8)
    else:
        compare(S, st, 1e-5, 1e-4)


@pytest.mark.parametrize("ndim,n", [(2, [24, 20]), (3, [12, 11, 10])])
def test_failed_cell_on_a_metric_without_atmosphere(G, ndim, n):
    """An energy below the field's own has no root: both sides count the failure, keep the cell's
    primitives and step on."""
    pr = P.random_box(22, ndim, n, metric=True)
    st = oracle.from_problem(pr)
    S = G.Solver.from_problem(pr)
    at = tuple(0 if k == 1 else k // 2 for k in S.shape)
    st.q[4][at] = -50.0
    S.q[4][at] = -50.0
    dt = S.compute_dt()
    st.step(dt)
    S.step(dt)
    assert st.fails > 0 and S.diagnostics()[2] == st.fails
    compare(S, st, 1e-10, 1e-8)
