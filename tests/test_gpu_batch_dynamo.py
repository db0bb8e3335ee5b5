"""A batch that holds problems with and without the mean-field dynamo (they take separate kernels
of the implicit solve): each is bitwise what it is in a batch of its own."""
import pytest

from paper_2110_03732_gb300 import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_dynamo_and_plain_problems_in_one_batch(precision):
    from paper_2110_03732_gb300 import build, grmhd
    build.build()
    probs = [P.dynamo_1d(n=37), P.orszag_tang(24), P.random_box(3, 2, [21, 18], xi=0.3, metric=True),
             P.random_box(4, 2, [19, 16], metric=True), P.random_box(5, 3, [9, 8, 7], xi=-0.2)]
    mixed, alone = ([grmhd.Solver.from_problem(p, precision=precision) for p in probs] for _ in range(2))
    dts = [s.compute_dt() for s in alone]
    B = grmhd.Batch(mixed)
    B.set_dt(dts)
    for s, dt in zip(alone, dts):
        b = grmhd.Batch([s])
        b.set_dt([dt])
        for _ in range(2):
            b.step()
    for _ in range(2):
        B.step()
    torch.cuda.synchronize()
    for k, (a, s) in enumerate(zip(alone, mixed)):
        assert torch.equal(a.state, s.state), k
        assert torch.isfinite(a.state).all()
