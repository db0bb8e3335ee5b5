"""The fixed-point MC and PPM cells of the FP64 reconstruction (csrc/fixrec.cuh), compiled
for the host and compared with exact rational arithmetic.

Tolerances (u = 2^-53, the rounding of one result; E the window's largest exponent, with a
last place of 2^-61 of its value range):
  * MC, every value within 2^7 of the largest: the correctly rounded states, exactly.
  * MC, any window: a saturated neighbour lies 2^5 above the larger of the two others, so a
    dropped bit is at most 2^-54 of max(|b|, |h|); three of them and the rounding stay
    within 4 u max(|b|, |h|).
  * PPM: at most eight dropped bits, 2^-56 of the window's largest value, and the rounding.
"""
import random
import shutil
import subprocess
from fractions import Fraction as Fr
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2110_03732_gb300" / "csrc"

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "fixrec.cuh"
using namespace grmhd;
int main() {
    char k;
    double v[6];
    while (std::scanf(" %c %la %la %la %la %la", &k, v, v + 1, v + 2, v + 3, v + 4) == 6) {
        double lo = 0, hi = 0, in = 0, s1 = 0;
        const bool ok = k == 'm' ? fx_mc_cell(v[0], v[1], v[2], lo, hi)
                                 : fx_ppm_cell(v[0], v[1], v[2], v[3], v[4], lo, hi, in, s1);
        std::printf("%d %a %a %a %a\n", (int)ok, lo, hi, in, s1);
    }
}
"""


@pytest.fixture(scope="module")
def cells(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fixrec")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-x", "c++", "-I", str(CSRC), str(d / "t.cpp"), "-o", str(d / "t")],
                   check=True)

    def run(kind, rows):
        text = "\n".join(kind + " " + " ".join(float(x).hex() for x in (list(r) + [0.0] * 5)[:5]) for r in rows)
        out = subprocess.run([str(d / "t")], input=text + "\n", capture_output=True, text=True, check=True).stdout
        return [(int(w[0]), [float.fromhex(x) for x in w[1:]]) for w in (ln.split() for ln in out.splitlines())]

    return run


def half_slope(a, b, x):
    d, c, e = b - a, (x - a) / 4, x - b
    if d > 0 and e > 0:
        return min(d, c, e)
    return max(d, c, e) if d < 0 and e < 0 else Fr(0)


def nearest(f):
    """The double nearest to a rational (Python's division rounds correctly)."""
    return f.numerator / f.denominator


def spread(vals):
    e = [abs(v) for v in vals if v]
    return max(e) / min(e) if e else 1.0


def windows(kind, n):
    rng = random.Random(3)
    out = []
    for _ in range(n):
        scale = 2.0 ** rng.uniform(-300, 300)
        base = rng.choice([0.0, 1.0, rng.uniform(-1, 1)])
        amp = 10.0 ** -rng.uniform(0, 12)
        if kind == "smooth":
            w = [scale * (base + amp * rng.uniform(-1, 1)) for _ in range(3)]
        elif kind == "jump":   # values of very different size, both signs, zeros
            w = [scale * rng.choice([-1, 1]) * rng.choice([0.0, 1.0, 2.0 ** -rng.uniform(0, 90)]) * rng.uniform(.5, 1)
                 for _ in range(3)]
        else:                  # equal values, ties and exact powers of two
            w = [scale * rng.choice([-1.0, -0.5, 0.0, 0.25, 0.5, 1.0, 1.5, 1.0 + 2.0 ** -52]) for _ in range(3)]
        out.append(w)
    return out


@pytest.mark.parametrize("kind", ["smooth", "jump", "ties"])
def test_mc_cell(cells, kind):
    rows = windows(kind, 4000)
    exact = 0
    for (a, b, x), (ok, (lo, hi, _, _)) in zip(rows, cells("m", rows)):
        assert ok
        fa, fb, fx = Fr(a), Fr(b), Fr(x)
        h = half_slope(fa, fb, fx)
        if spread([a, b, x]) < 2 ** 7:
            exact += 1
            assert (lo, hi) == (nearest(fb - h), nearest(fb + h))
        tol = Fr(4, 2 ** 53) * max(abs(fb), abs(h))
        assert abs(Fr(lo) - (fb - h)) <= tol and abs(Fr(hi) - (fb + h)) <= tol
        if h == 0:
            assert lo == b and hi == b
    assert exact > 100


@pytest.mark.parametrize("bad", [float("inf"), -float("inf"), float("nan"), 1e-300])
def test_mc_cell_refuses(cells, bad):
    """Non-finite windows, and nonzero ones below 2^-943, go to the FP64 sequence; a window
    of zeros does not."""
    rows = [[bad, 1.0, 2.0], [1.0, bad, 2.0], [1.0, 2.0, bad]] if abs(bad) != 1e-300 else [[bad, 2 * bad, 0.0]]
    assert all(ok == 0 for ok, _ in cells("m", rows))
    assert cells("m", [[0.0, -0.0, 0.0]]) == [(1, [0.0, 0.0, 0.0, 0.0])]


@pytest.mark.parametrize("kind", ["smooth", "ties"])
def test_ppm_cell(cells, kind):
    rng = random.Random(5)
    rows = []
    for w in windows(kind, 4000):
        a0, a1, x = w
        s0 = (a1 - a0) * rng.choice([0.0, 0.3, 1.0, 2.0])
        rows.append([a0, a1, x, s0, a0 - (a1 - a0) * rng.uniform(-1, 1)])
    used = 0
    for r, (ok, (lo, hi, ins, s1)) in zip(rows, cells("p", rows)):
        if spread(r[:3]) < 2 ** 6 and spread(r[:3] + [max(map(abs, r))]) < 2 ** 6:
            assert ok
        if not ok:
            continue
        used += 1
        a0, a1, x, s0, ip = map(Fr, r)
        fs1 = 2 * half_slope(a0, a1, x)
        fin = a0 + (a1 - a0) / 2 - (fs1 - s0) / 6
        l, rr = ip, fin
        if (rr - a0) * (a0 - l) <= 0:
            l = rr = a0
        else:
            dd, m6 = rr - l, 6 * (a0 - (l + rr) / 2)
            if dd * m6 > dd * dd:
                l = 3 * a0 - 2 * rr
            elif -dd * dd > dd * m6:
                rr = 3 * a0 - 2 * l
        big = Fr(1, 2 ** 56) * max(abs(v) for v in (a0, a1, x, s0, ip))
        for got, want in ((lo, l), (hi, rr), (ins, fin), (s1, fs1)):
            assert abs(Fr(got) - want) <= abs(want) / 2 ** 53 + big
    assert used > 1000


@pytest.mark.parametrize("far", [0.0, 1e-290, 1.0, -1e200])
def test_mc_cell_of_tiny_values(cells, far):
    """Where the two smaller values lie below 2^-943 the cell goes to the FP64 sequence, however
    large the third is; so whatever is accepted keeps the bound of any window.  Denormals count
    as zero: a cell of which one difference is then zero is flat, off by no more than 2^-1022."""
    rng = random.Random(7)
    tiny = [0.0, 5e-324, 1e-310, 3e-308, 1e-300, 2e-300, 1e-286]
    rows = []
    for _ in range(600):
        w = [far, rng.choice([-1, 1]) * rng.choice(tiny), rng.choice([-1, 1]) * rng.choice(tiny)]
        rng.shuffle(w)
        rows.append(w)
    for (a, b, x), (ok, (lo, hi, _, _)) in zip(rows, cells("m", rows)):
        if not ok:
            continue
        fb = Fr(b)
        h = half_slope(Fr(a), fb, Fr(x))
        tol = Fr(4, 2 ** 53) * max(abs(fb), abs(h)) + Fr(1, 2 ** 1022)
        assert abs(Fr(lo) - (fb - h)) <= tol and abs(Fr(hi) - (fb + h)) <= tol
    flat = [[0.0, 0.0, far], [far, 0.0, 0.0], [0.0, 0.0, 0.0]]
    assert cells("m", flat) == [(1, [0.0] * 4)] * 3
