"""The float64 window table on the host: its polynomials, and what a new window costs."""
import math
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2302_00414_gb300", "csrc")

PROGRAM = r"""
#include "polytable.h"
#include <chrono>
#include <cstdio>
#include <cstdlib>
using namespace infft;
int main(int argc, char** argv) {
    const int m = atoi(argv[1]);
    const double beta = atof(argv[2]);
    std::vector<double> c;
    kb_poly_table<22>(m, beta, m, c);
    double best = 1e9;
    for (int r = 0; r < 30; ++r) {
        const auto t0 = std::chrono::steady_clock::now();
        kb_poly_table<22>(m, beta * (1.0 - 1e-3 * r), m, c);
        best = std::min(best, std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count());
    }
    kb_poly_table<22>(m, beta, m, c);
    printf("%.9g\n", best);
    for (double v : c) printf("%.17g\n", v);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("poly")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run([cc, "-O2", "-std=c++17", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    return str(d / "t")


def _run(program, m, beta):
    out = subprocess.run([program, str(m), repr(beta)], capture_output=True, text=True, check=True).stdout.split()
    return float(out[0]), [float(v) for v in out[1:]]


@pytest.mark.parametrize("ratio", [1.0, 0.5, 0.375, 0.1])
@pytest.mark.parametrize("m", [1, 2, 4, 8, 15])
def test_coefficients_of_the_interpolant(program, m, ratio):
    """The coefficients are those of the polynomial through the window's values at the 22 nodes (in floating point the
    doubles nearest cos(pi (k + 1/2) / 22)), rounded once: half a unit of the last place each, and 1e-20 of
    the tap's largest for the double-doubles (1e-29 per value, multiplied by a change of basis below 1e8)."""
    mp = pytest.importorskip("mpmath")
    beta, n = math.pi * m * (2 - ratio), 22
    _, c = _run(program, m, beta)
    x = [math.cos(math.pi * (k + 0.5) / n) for k in range(n)]
    with mp.workdps(50):
        xs = [mp.mpf(v) for v in x]
        for s in sorted({1, (m + 1) // 2, m}):
            d = [mp.besseli(0, mp.mpf(beta) * mp.sqrt(max(mp.mpf(0), 1 - (((v + 1) / 2 + m - s) / m) ** 2))) for v in xs]
            for j in range(1, n):     # Newton's form, then powers
                for k in range(n - 1, j - 1, -1):
                    d[k] = (d[k] - d[k - 1]) / (xs[k] - xs[k - j])
            e = [mp.mpf(0)] * n
            for j in range(n - 1, -1, -1):
                for k in range(n - 1, 0, -1):
                    e[k] = e[k - 1] - e[k] * xs[j]
                e[0] = -e[0] * xs[j] + d[j]
            top = max(abs(v) for v in e)
            for k in range(n):
                assert abs(mp.mpf(c[k * m + s - 1]) - e[k]) <= abs(e[k]) * mp.mpf(2) ** -53 + top * mp.mpf("1e-20")


def test_cost_of_a_new_window(program):
    """A plan with a new window makes its table while the program waits: the best of 30 takes a fraction of the 0.4 ms
    that a small float64 plan takes besides."""
    assert _run(program, 8, 8 * math.pi * 1.5)[0] < 2.5e-4


SPLINE = r"""
#include "polytable.h"
#include <cstdio>
#include <cstdlib>
int main(int argc, char** argv) {
    std::vector<float> c;
    infft::bspline_poly_table<11>(atoi(argv[1]), 8, c);
    for (float v : c) printf("%.9g\n", v);
}
"""


@pytest.mark.parametrize("m", range(1, 9))
def test_float32_spline_table(m, tmp_path):
    """The polynomials against the B-spline in rational arithmetic: the coefficients' float32 rounding, half a unit each
    (the constant's low part is in the table), and 1e-11 of the largest value for order 16 in degree 10."""
    from fractions import Fraction
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host compiler")
    (tmp_path / "s.cpp").write_text(SPLINE)
    subprocess.run([cc, "-O2", "-std=c++17", "-I", CSRC, str(tmp_path / "s.cpp"), "-o", str(tmp_path / "s")], check=True)
    out = subprocess.run([str(tmp_path / "s"), str(m)], capture_output=True, text=True, check=True).stdout.split()
    c = [float(v) for v in out]
    n = 2 * m
    for s in range(1, m + 1):
        col = [c[8 * k + s - 1] for k in range(12)]
        bound = 2.0 ** -24 * sum(abs(v) for v in col[1:11]) + 2.0 ** -47 * abs(col[0]) + 1e-11
        for u in (Fraction(0), Fraction(1, 7), Fraction(1, 2), Fraction(15, 16), Fraction(1)):
            y = u + m - s + Fraction(n, 2)
            ref = sum((-1) ** k * math.comb(n, k) * (y - k) ** (n - 1) for k in range(n + 1) if y > k) / math.factorial(n - 1)
            v = 2 * u - 1
            p = sum(Fraction(col[k]) * v ** k for k in range(11)) + Fraction(col[11])
            assert abs(float(p - ref)) <= bound
